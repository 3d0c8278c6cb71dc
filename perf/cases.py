"""The library's work as its users have it done, for timing.

Three kinds of pass, each through the public calls of
``paper_0707_2437_gb300/lbm.py``, with the fields on the GPU:

* ``job``     one grid: ``init`` from (rho, ux, uy), ``step(n)``, ``moments``;
* ``series``  one grid measured while it runs, as in the sound-speed and
              viscosity fits: ``init``, then ``step(every)`` and ``mode`` in
              turn, ``sums`` and ``moments`` at the end;
* ``batch``   many grids: ``init`` of each, one ``Batch.step`` for all of them
              (lockstep, or the flow schedule with a step limit per grid, as
              the server calls it), ``moments`` of each.

The grids, the batch, the c2 field and the output arrays are made once in
``prepare``, as a program keeps them.  Every pass starts with ``init``, so a
pass can be repeated and gives the same outputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0707_2437_gb300 import lbm

# Floating-point operations of one lattice update (Eq. 5): density 11, momentum
# and velocity 14, the shared equilibrium and force terms 20, nine outputs 44.
FLOPS_PER_UPDATE = 89
# Most lattice updates of a drawn case (the listed sweep makes 3.8e9).
MOST_UPDATES = 3.0e9


def _job(name, nx, ny, storage, tau, c2, amp, steps, lens=False, drive=0.0, period=500.0):
    return {"name": name, "kind": "job", "nx": nx, "ny": ny, "storage": storage, "tau": tau,
            "c2": c2, "amp": amp, "steps": steps, "lens": lens, "drive": drive,
            "period": period}


def listed():
    return [
        # The viscous-decay run of the paper's Fig. 6 (alpha = -0.6, lambda =
        # 400, four rows): ten of its hundred periods.  The smallest grid in
        # use; a step is far below a launch.
        _job("decay_400x4_f32", 400, 4, "f32", 0.55, 1 / 3 + 0.6, 1e-3, 4140),
        # A sound-speed measurement on a 512 x 4 standing wave in FP16 storage:
        # the density mode is read every 1/60 period.
        {"name": "speed_512x4_f16d", "kind": "series", "nx": 512, "ny": 4, "storage": "f16d",
         "tau": 0.6, "c2": 0.15, "amp": 1e-3, "every": 22, "reads": 120},
        # The driven channel of the paper's Fig. 1: a boundary update each step.
        _job("driven_8192x4_f32", 8192, 4, "f32", 0.53, 0.3333, 1e-4, 1000, drive=1e-4),
        # A ragged domain: odd in both directions, no vector width divides it.
        _job("odd_509x381_f32", 509, 381, "f32", 0.7, 0.25, 1e-3, 500),
        # An ordinary FP32 grid whose state stays in the L2 cache.
        _job("grid_1024_f32", 1024, 1024, "f32", 0.8, 0.2, 1e-3, 512),
        # A per-site sound speed (an acoustic lens) on a large FP32 grid.
        _job("lens_2048_f32", 2048, 2048, "f32", 0.8, 0.2, 5e-3, 100, lens=True),
        # BF16 storage with stochastic rounding, the unbiased 16-bit form.
        _job("stochastic_2048_bf16d", 2048, 2048, "bf16d-sr", 0.9, 0.15, 1e-3, 200),
        # The largest configured grid: 8192^2 with Fourier modes, FP16 storage.
        _job("fourier_8192_f16d", 8192, 8192, "f16d", 0.6, 0.15, 1e-3, 50),
        # The parameter sweep: nine 2048^2 grids stepped together, FP32.
        {"name": "sweep_9x2048_f32", "kind": "batch", "count": 9, "lo": 2048, "hi": 2048,
         "aspect": 0.0, "storage": "f32", "schedule": "lockstep", "steps": 100, "sizes": 1},
        # The same sweep in FP16 storage, the throughput form.
        {"name": "sweep_9x2048_f16d", "kind": "batch", "count": 9, "lo": 2048, "hi": 2048,
         "aspect": 0.0, "storage": "f16d", "schedule": "lockstep", "steps": 100, "sizes": 1},
        # Many uneven grids, half FP32 and half FP16, in one lockstep batch.
        {"name": "uneven_192_mixed", "kind": "batch", "count": 192, "lo": 64, "hi": 1024,
         "aspect": 2.0, "storage": "mixed", "schedule": "lockstep", "steps": 100, "sizes": 4},
        # One launch of the server below capacity: the flow schedule with a
        # share of 1e9 updates for each resident grid.
        {"name": "serve_20_flow_mixed", "kind": "batch", "count": 20, "lo": 128, "hi": 2048,
         "aspect": 1.0, "storage": "mixed", "schedule": "flow", "steps": 1024, "sizes": 5},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def width(lo, hi):
        n = log_int(lo, hi)
        return max(8, (n + 4) // 8 * 8) if rng.random() < 0.6 else n

    storages = ["f32", "f32", "f16d", "bf16d", "f16d-sr", "bf16d-sr"]
    tau = round(rng.uniform(0.55, 1.5), 4)
    c2 = round(rng.uniform(0.05, 0.45), 4)
    amp = round(math.exp(rng.uniform(math.log(1e-3), math.log(2e-2))), 6)
    kind = rng.choice(["job", "job", "job", "series", "batch", "batch"])
    if kind == "batch":
        hi = rng.choice([256, 512, 1024, 2048])
        lo = rng.choice([64, 128, hi])
        count = log_int(2, 128)
        count = max(1, min(count, int(MOST_UPDATES / (hi * hi * 20))))
        schedule = rng.choice(["lockstep", "lockstep", "flow"])
        steps = log_int(20, 400)
        steps = max(10, min(steps, int(MOST_UPDATES / (count * hi * hi))))
        return {"kind": "batch", "count": count, "lo": lo, "hi": hi,
                "aspect": rng.choice([0.0, 1.0, 2.0]),
                "storage": rng.choice(["f32", "f16d", "bf16d", "f16d-sr", "mixed"]),
                "schedule": schedule, "steps": steps, "sizes": rng.randrange(1 << 20)}
    nx, ny = width(64, 4096), width(4, 4096)
    # The shortest wave keeps a good part of its amplitude.
    k2 = (max(1, _most_waves(nx)) / nx) ** 2 + (_most_waves(ny) / ny) ** 2
    lasts = int(1.5 / ((2 * tau - 1) / 6 * 4 * math.pi ** 2 * k2))
    if kind == "series":
        reads = log_int(10, 60)
        every = log_int(2, 40)
        every = max(1, min(every, int(MOST_UPDATES / (4 * reads * nx * ny)), lasts // reads))
        return {"kind": "series", "nx": nx, "ny": ny, "storage": rng.choice(storages),
                "tau": tau, "c2": c2, "amp": amp, "every": every, "reads": reads}
    steps = max(4, min(log_int(30, 3000), int(MOST_UPDATES / (nx * ny)), lasts))
    case = _job("", nx, ny, rng.choice(storages), tau, c2, amp, steps)
    option = rng.random()
    if option < 0.2 and not case["storage"].endswith("-sr"):
        case["lens"] = True
    elif option > 0.85:
        case["drive"] = 1e-3
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# Inputs.

def _grids(case):
    """The grids of a case: dicts of nx, ny, storage, tau, c2, amp, steps."""
    if case["kind"] != "batch":
        steps = case["steps"] if case["kind"] == "job" else case["every"] * case["reads"]
        return [{"nx": case["nx"], "ny": case["ny"], "storage": case["storage"],
                 "tau": case["tau"], "c2": case["c2"], "amp": case["amp"], "steps": steps}]
    rng = np.random.default_rng(case["sizes"])
    out = []
    for j in range(case["count"]):
        sites = math.exp(rng.uniform(math.log(case["lo"] ** 2), math.log(case["hi"] ** 2)))
        aspect = 2.0 ** rng.uniform(-case["aspect"], case["aspect"])
        nx = max(8, int(round(math.sqrt(sites * aspect) / 8)) * 8)
        ny = max(8, int(round(math.sqrt(sites / aspect) / 8)) * 8)
        storage = case["storage"]
        if storage == "mixed":
            storage = "f32" if rng.random() < 0.5 else "f16d"
        out.append({"nx": nx, "ny": ny, "storage": storage,
                    "tau": float(rng.uniform(0.55, 1.2)), "c2": float(rng.uniform(0.05, 0.4)),
                    "amp": float(np.exp(rng.uniform(np.log(1e-3), np.log(2e-2)))),
                    "steps": case["steps"]})
    if case["schedule"] == "flow":
        # The server's shares: updates in proportion to the square root of the
        # sites, 1e9 for the whole launch, at most `steps` steps a grid.
        total = sum(math.sqrt(g["nx"] * g["ny"]) for g in out)
        for g in out:
            share = 1.0e9 * math.sqrt(g["nx"] * g["ny"]) / total
            g["steps"] = max(1, min(case["steps"], int(share / (g["nx"] * g["ny"]))))
    return out


def _most_waves(n):
    """Largest wave number of the inputs along a side of n sites: waves are long
    against the lattice, as in every run of the paper, and thin channels carry
    plane waves."""
    return min(4, n // 128) if n >= 128 else int(n >= 64)


def _fields(nx, ny, amp, rng, device):
    """rho, ux, uy: a rest fluid of unit density with eight plane waves of the
    given density amplitude and slow flow of a few plane waves."""
    mx, my = max(1, _most_waves(nx)), _most_waves(ny)
    x = torch.arange(nx, dtype=torch.float64, device=device)[None, :] * (2 * math.pi / nx)
    y = torch.arange(ny, dtype=torch.float64, device=device)[:, None] * (2 * math.pi / ny)

    def waves(count, a):
        w = rng.uniform(0.5, 1.0, count)
        w *= a / w.sum()
        out = torch.zeros(ny, nx, dtype=torch.float64, device=device)
        for j in range(count):
            kx, ky = 0, 0
            while kx == 0 and ky == 0:
                kx, ky = int(rng.integers(-mx, mx + 1)), int(rng.integers(-my, my + 1))
            p = rng.uniform(0, 2 * math.pi)
            # cos(a + b) from the two one-dimensional factors
            out += w[j] * (torch.cos(kx * x) * torch.cos(ky * y + p)
                           - torch.sin(kx * x) * torch.sin(ky * y + p))
        return out

    return 1.0 + waves(8, amp), waves(3, 0.3 * amp), waves(3, 0.3 * amp)


def _lens(nx, ny, c2, device):
    """c2 raised by half in a Gaussian bump at the centre (an acoustic lens)."""
    x = (torch.arange(nx, dtype=torch.float64, device=device)[None, :] + 0.5) / nx - 0.5
    y = (torch.arange(ny, dtype=torch.float64, device=device)[:, None] + 0.5) / ny - 0.5
    return c2 * (1.0 + 0.5 * torch.exp(-(x * x + y * y) / (2 * 0.15 ** 2)))


def _inputs(case, seed, device):
    rng = np.random.default_rng(seed)
    return [_fields(g["nx"], g["ny"], g["amp"], rng, device) for g in _grids(case)]


class _State:
    """What a program keeps between passes."""

    def __init__(self, case, seed):
        self.case = case
        self.plan = _grids(case)
        self.fields = _inputs(case, seed, "cuda")
        self.grids = []
        for g in self.plan:
            grid = lbm.Grid(g["nx"], g["ny"], g["tau"], g["c2"],
                            g["storage"].replace("-sr", ""))
            if g["storage"].endswith("-sr"):
                grid.set_rounding("stochastic")
            self.grids.append(grid)
        if case.get("lens"):
            self.grids[0].set_c2_field(_lens(case["nx"], case["ny"], case["c2"], "cuda"))
        if case.get("drive"):
            self.grids[0].set_drive(case["drive"], case["period"])
        # rho, ux, uy of all grids end to end in one array each, a view a grid.
        ends = np.cumsum([g["nx"] * g["ny"] for g in self.plan])
        self.out = [torch.empty(int(ends[-1]), dtype=torch.float64, device="cuda")
                    for _ in range(3)]
        self.views = []
        for g, end in zip(self.plan, ends):
            lo = int(end) - g["nx"] * g["ny"]
            self.views.append([o[lo:int(end)].view(g["ny"], g["nx"]) for o in self.out])
        self.batch = None
        if case["kind"] == "batch":
            self.batch = lbm.Batch(self.grids)
            if case["schedule"] == "flow":
                self.batch.set_schedule("flow")
            self.steps = max(g["steps"] for g in self.plan)
            self.limits = [g["steps"] for g in self.plan] if case["schedule"] == "flow" else None

    def __del__(self):
        if getattr(self, "batch", None) is not None:
            self.batch.close()
        for g in getattr(self, "grids", []):
            g.close()


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    for grid, fields in zip(state.grids, state.fields):
        grid.init(*fields)
    out = {}
    kind = state.case["kind"]
    if kind == "job":
        state.grids[0].step(state.case["steps"])
    elif kind == "series":
        grid, series = state.grids[0], []
        for _ in range(state.case["reads"]):
            grid.step(state.case["every"])
            series.append(grid.mode("rho", 1, 0))
        out["modes"] = np.stack(series)
        out["sums"] = grid.sums()
    else:
        state.batch.step(state.steps, state.limits)
        state.batch.sync()
    for grid, views in zip(state.grids, state.views):
        grid.moments(out=views)
    out["rho"], out["ux"], out["uy"] = state.out
    return out


def work(case):
    """The fields in and out (three doubles a site each way, and the c2 field),
    and the arithmetic of every lattice update."""
    sites = sum(g["nx"] * g["ny"] for g in _grids(case))
    updates = sum(g["nx"] * g["ny"] * g["steps"] for g in _grids(case))
    bytes_ = 48 * sites + (4 * sites if case.get("lens") else 0)
    return {"bytes": bytes_, "flops": FLOPS_PER_UPDATE * updates}


# ---------------------------------------------------------------------------
# The same update in 64 bits, written out from the paper.

_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _equilibrium(rho, ux, uy, out):
    usq = 1.0 - 1.5 * (ux * ux + uy * uy)
    for i in range(9):
        eu = _EX[i] * ux + _EY[i] * uy
        torch.mul(_W[i] * rho, usq + 3.0 * eu + 4.5 * eu * eu, out=out[i])
    return out


def _moments(f):
    rho = f.sum(0)
    ux = (f[1] + f[5] + f[8] - f[3] - f[6] - f[7]) / rho
    uy = (f[2] + f[5] + f[6] - f[4] - f[7] - f[8]) / rho
    return rho, ux, uy


def _step(f, feq, tau, alpha, drive=None):
    """Collide (Eq. 2 and 5, central differences) and stream, in place."""
    rho, ux, uy = _moments(f)
    gx = 1.5 * alpha * (torch.roll(rho, -1, 1) - torch.roll(rho, 1, 1))
    gy = 1.5 * alpha * (torch.roll(rho, -1, 0) - torch.roll(rho, 1, 0))
    _equilibrium(rho, ux, uy, feq)
    f.lerp_(feq, 1.0 / tau)
    for i in range(9):
        if i:
            f[i] += _W[i] * (_EX[i] * gx + _EY[i] * gy)
        if drive is not None:  # equilibrium columns at rest
            f[i, :, 0] = _W[i] * drive
            f[i, :, -2:] = _W[i]
        if i:
            f[i] = torch.roll(f[i], (_EY[i], _EX[i]), (0, 1))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    plan, out, modes = _grids(case), [[], [], []], []
    rng = np.random.default_rng(seed)
    for g in plan:
        nx, ny = g["nx"], g["ny"]
        fields = _fields(nx, ny, g["amp"], rng, dev)
        f = _equilibrium(*fields, torch.empty(9, ny, nx, dtype=torch.float64, device=dev))
        feq = torch.empty_like(f)
        alpha = 1 / 3 - (_lens(nx, ny, g["c2"], dev) if case.get("lens") else g["c2"])
        px = torch.arange(nx, dtype=torch.float64, device=dev) * (2 * math.pi / nx)
        wave = torch.stack([torch.cos(px), torch.sin(px)]) * (2.0 / (nx * ny))
        for t in range(g["steps"]):
            drive = None
            if case.get("drive"):
                drive = 1.0 + case["drive"] * math.sin(2 * math.pi * t / case["period"])
            _step(f, feq, g["tau"], alpha, drive)
            if case["kind"] == "series" and (t + 1) % case["every"] == 0:
                modes.append((wave * (f.sum(0) - 1.0).sum(0)).sum(1))
        rho, ux, uy = _moments(f)
        for o, v in zip(out, (rho, ux, uy)):
            o.append(v.reshape(-1))
        if case["kind"] == "series":
            sums = torch.stack([rho.sum(), (rho * ux).sum(), (rho * uy).sum()])
    rho, ux, uy = (torch.cat(o) for o in out)
    answer = {"rho": rho, "ux": ux, "uy": uy}
    if case["kind"] == "series":
        answer["modes"] = torch.stack(modes).cpu().numpy()
        answer["sums"] = sums.cpu().numpy()
    return answer

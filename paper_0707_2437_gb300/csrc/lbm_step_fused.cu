// The single-grid step kernel that advances two or three time steps per launch
// (the fused walk of lbm_fused.cuh), and the plan that sizes its tiles.
#include "lbm_internal.h"
#include "lbm_launch.cuh"
#include "lbm_fused.cuh"

namespace vss {

namespace {

constexpr int kWarps = 4;  // warps per block

// Bound: HBM for FP32 with two steps, shared memory and issue with three; instruction
// issue for the 16-bit kinds.  Eight warps per SM of up to 255 registers, with two
// rows of copies in flight each: twelve warps at 168 registers, with the first
// stage's waiting row in shared memory too, spent the time on shared-memory traffic
// in FP32 (71 % of its bandwidth; 8192^2 158k against 172k MLUPS) and spilled in the
// 16-bit kinds (214k against 245k).  Measured on one grid, per step, single steps
// before and passes now: 8192^2 FP32 705.7 -> 354 us (190k MLUPS; 24 B an update),
// FP16 372.5 -> 271 us (248k), BF16 with stochastic rounding 371.0 -> 295; 4096^2 FP32
// 185 -> 89.8, FP16 107 -> 71.7; 2048^2 FP32 49.6 -> 26.3, FP16 25.3 -> 23.5, FP32 with
// a c2 field 54.0 -> 29.8.  RAG (rows copied and stored word by word, coalesced, which
// adds a staging row and some 100 of 1200 instructions a row step): 2002 x 2004 FP32
// 49.5 -> 36.5, FP16 35.2 -> 28.2.
template <int S, int RND, int VA, int TS, bool RAG>
__global__ void __launch_bounds__(32 * kWarps, 2)
    k_step_fused(const void *__restrict__ fin, void *__restrict__ fout, int nx, int ny, size_t P,
                 FusedStrips strips, long long ntiles, int rows, Coef c, int steps, const uint32_t *tdev,
                 uint32_t toff, const float *__restrict__ a15f) {
    extern __shared__ uint4 walk_smem[];
    pdl_enter();
    const long long tile = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (tile >= ntiles) return;  // whole warps leave together
    constexpr bool PACK = fused_packs(S) && !RAG;
    // Whole strips segment by segment, then the packed tiles.
    const long long whole = (long long)strips.full * ((ny + rows - 1) / rows);
    int seg, x0, y0, y1, lanes = 32;
    if (!PACK || tile < whole) {
        seg = (int)(tile / strips.full);
        x0 = (int)(tile - (long long)seg * strips.full) * FusedGeom<S, TS>::COLS;
        y0 = seg * rows;
        y1 = min(ny, y0 + rows);
    } else {
        seg = (int)(tile - whole);
        x0 = strips.full * FusedGeom<S, TS>::COLS;
        y0 = seg * strips.pieces * rows;
        y1 = min(ny, y0 + strips.pieces * rows);
        lanes = strips.lanes;
    }
    const int high = min(rows, y1 - y0);
    FusedWalk<S, LD_NC, RND, VA, TS, PACK, RAG> w(fin, fout, nx, ny, P, x0, y0, y1, high,
                                                  PACK ? lanes : 32);
    if constexpr (VA) w.a15f = a15f;
    if constexpr (RND) w.set_step((tdev ? *tdev : 0u) + toff);
    // Neighbouring segments walk in opposite directions, so the rows they
    // share are read by both at about the same time.
    w.run(high, (seg & 1) ? -1 : 1, steps, c,
          walk_smem + (threadIdx.x >> 5) * fused_vecs<S, VA, TS, RAG>());
}

using FusedKernel = void (*)(const void *, void *, int, int, size_t, FusedStrips, long long, int,
                             Coef, int, const uint32_t *, uint32_t, const float *);

struct Choice {
    FusedKernel fn = nullptr;
    int smem = 0;
};

template <int S, int RND, int VA, int TS, bool RAG = false>
Choice choice() {
    return Choice{k_step_fused<S, RND, VA, TS, RAG>, kWarps * fused_vecs<S, VA, TS, RAG>() * 16};
}

// The kernel for widths that are no multiple of the lanes' vectors (two steps).
Choice choose_ragged(int storage, int rnd) {
    switch (storage) {
        case ST_F32: return choice<ST_F32, 0, 0, 2, true>();
        case ST_F16: return rnd ? choice<ST_F16, 1, 0, 2, true>() : choice<ST_F16, 0, 0, 2, true>();
        case ST_BF16:
            return rnd ? choice<ST_BF16, 1, 0, 2, true>() : choice<ST_BF16, 0, 0, 2, true>();
        default: return Choice{};
    }
}

Choice choose(int storage, int rnd, bool field, int steps) {
    switch (storage) {
        case ST_F32:
            if (field) return steps == 3 ? choice<ST_F32, 0, 1, 3>() : choice<ST_F32, 0, 1, 2>();
            return steps == 3 ? choice<ST_F32, 0, 0, 3>() : choice<ST_F32, 0, 0, 2>();
        case ST_F16:
            return field ? choice<ST_F16, 0, 1, 2>()
                         : (rnd ? choice<ST_F16, 1, 0, 2>() : choice<ST_F16, 0, 0, 2>());
        case ST_BF16:
            return field ? choice<ST_BF16, 0, 1, 2>()
                         : (rnd ? choice<ST_BF16, 1, 0, 2>() : choice<ST_BF16, 0, 0, 2>());
        default:
            return Choice{};
    }
}

}  // namespace

Err plan_fused(int storage, int rnd, bool field, int nx, int ny, FusedPlan *out) {
    *out = FusedPlan{};
    const bool ragged = nx % fused_vec(storage) != 0;
    if (!fused_width(storage, nx) || (field && (rnd || ragged))) return cudaSuccess;
    double best = 1e30;
    for (int steps = 2; steps <= (ragged ? 2 : fused_most_steps(storage)); ++steps) {
        const Choice ch = ragged ? choose_ragged(storage, rnd)
                                 : choose(storage, rnd, field, steps);
        const long long wave = resident_warps((const void *)ch.fn, kWarps, ch.smem);
        if (wave <= 0) return cudaErrorLaunchOutOfResources;
        const FusedStrips strips = fused_strips(storage, steps, nx);
        // Tile height: a tile costs some row steps beyond its rows, and a launch
        // lasts as many tiles as its fullest warp slot runs.
        const int most = fused_most_rows(storage, steps);
        long long least = -1;
        int rows = 2;
        for (int r = 2; r <= most; ++r) {
            const long long tiles = strips.tiles((ny + r - 1) / r);
            const long long cost = ((tiles + wave - 1) / wave) * (r + fused_overhead(steps));
            if (least < 0 || cost < least) {
                least = cost;
                rows = r;
            }
            if (r >= ny) break;
        }
        // A row step of three steps takes about 1.22 times as long as one of two, 1.3
        // times with a c2 field (three steps against two: 1024^2 10.42 / 9.84 us a
        // step, 1536^2 19.2 / 18.4, 2048^2 29.9 / 31.2, 4096^2 102.4 / 114.3, 8192^2
        // 406 / 414).
        const double per_step =
            (double)least / (steps == 3 ? 3 / (field ? 1.3 : 1.22) : 2.0);
        if (per_step >= best) continue;
        best = per_step;
        out->steps = steps;
        out->rows = rows;
        out->strips = strips;
        out->ntiles = strips.tiles((ny + rows - 1) / rows);
    }
    // Passes or single steps: short tiles repeat much of the earlier steps' work, and a
    // launch lasts one walk of some rows however small the grid.  Estimates in
    // microseconds per step: row_us a row step of two steps in the fullest warp slot,
    // halved; a single step takes `even` a million sites, and `idle` more for every
    // site's worth of lanes beyond the width in its strips.  Measured per step, single
    // steps / passes: FP32 768^2 7.16 / 7.15, 1024^2 10.97 / 9.46, 2048^2 49.6 / 26.2,
    // 124 x 9600 11.4 / 14.8, 244 x 4800 11.1 / 11.8, 248 x 9600 27.1 / 20.4; with a
    // c2 field 768^2 6.9 / 7.5, 1024^2 11.75 / 9.86, 16 x 100000 54.6 / 60.5; FP16
    // 1024^2 8.85 / 10.4, 1536^2 15.2 / 15.1, 2048^2 25.3 / 23.5, 136 x 12000 20.7 /
    // 16.0, 64 x 40000 53.8 / 17.2; with stochastic rounding, whose conversion is the
    // slower for FP16, BF16 1536^2 16.9 / 16.2, 2048^2 27.6 / 25.3, FP16 2048^2 26.7 /
    // 27.1, 2048 x 4096 55.1 / 47.4.  Without 16-byte lanes both move words: FP32 1022
    // x 1024 11.2 / 12.1, 1202 x 1200 16.8 / 15.2, 242 x 4800 12.7 / 16.1, 2002 x 2004
    // 49.5 / 36.5, 8002 x 8000 730 / 491; FP16 1302 x 1300 15.0 / 15.5, 1402 x 1400
    // 16.3 / 15.6, 1446 x 1440 16.3 / 18.5, 2002 x 2004 35.2 / 28.2, 8002 x 8000 509 /
    // 347; BF16 with stochastic rounding 2002 x 2004 36.7 / 30.4, FP16 37.2 / 31.7.
    const bool wide = storage == ST_F32, slow = rnd && storage == ST_F16;
    double row_us, even, idle;
    int strip;  // columns of a single step's strips
    if (ragged) {
        row_us = wide ? 2.0 : rnd ? (slow ? 3.0 : 2.82) : 2.6;
        even = wide ? 11.4 : rnd ? 9.0 : 8.5;
        idle = 0;
        strip = 32;
    } else if (wide) {
        row_us = 1.43;
        even = field ? 11.2 : 9.6;
        idle = field ? 7.0 : 4.0;
        strip = field ? 64 : 128;
    } else {
        row_us = field ? 2.3 : rnd ? (slow ? 2.58 : 2.41) : 2.2;
        even = field ? 7.0 : rnd ? (slow ? 6.4 : 7.2) : 5.8;
        idle = 5.3;
        strip = field ? 128 : 256;
    }
    const double lanes = (double)((nx + strip - 1) / strip) * strip / nx;
    out->ok = best * row_us < 1e-6 * nx * ny * (even + idle * (lanes - 1));
    return cudaSuccess;
}

Err launch_fused(const FusedPlan &p, int storage, const void *fin, void *fout, int nx, int ny,
                 size_t P, const Coef &c, int steps, int rnd, const uint32_t *tdev, uint32_t toff,
                 const float *a15f, cudaStream_t st) {
    if (!p.ok) return cudaErrorInvalidValue;
    const Choice ch = nx % fused_vec(storage) ? choose_ragged(storage, rnd)
                                              : choose(storage, rnd, a15f != nullptr, p.steps);
    return launch_pdl(ch.fn, (unsigned)((p.ntiles + kWarps - 1) / kWarps), 32u * kWarps,
                      (size_t)ch.smem, st, fin, fout, nx, ny, P, p.strips, p.ntiles, p.rows, c,
                      steps, tdev, toff, a15f);
}

}  // namespace vss

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
// before and passes now: 8192^2 FP32 705.7 -> 353 us (190k MLUPS; 24 B an update),
// FP16 372.5 -> 274 us (245k), BF16 with stochastic rounding 371.0 -> 297; 4096^2 FP32
// 185 -> 89.7; 2048^2 FP32 49.6 -> 26.3, FP16 25.3 -> 23.4, FP32 with a c2 field 54.0
// -> 31.1.
template <int S, int RND, int VA, int TS>
__global__ void __launch_bounds__(32 * kWarps, 2)
    k_step_fused(const void *__restrict__ fin, void *__restrict__ fout, int nx, int ny, size_t P,
                 FusedStrips strips, long long ntiles, int rows, Coef c, int steps, const uint32_t *tdev,
                 uint32_t toff, const float *__restrict__ a15f) {
    extern __shared__ uint4 walk_smem[];
    pdl_enter();
    const long long tile = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (tile >= ntiles) return;  // whole warps leave together
    constexpr bool PACK = fused_packs(S);
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
    FusedWalk<S, LD_NC, RND, VA, TS, PACK> w(fin, fout, nx, ny, P, x0, y0, y1, high,
                                             PACK ? lanes : 32);
    if constexpr (VA) w.a15f = a15f;
    if constexpr (RND) w.set_step((tdev ? *tdev : 0u) + toff);
    // Neighbouring segments walk in opposite directions, so the rows they
    // share are read by both at about the same time.
    w.run(high, (seg & 1) ? -1 : 1, steps, c,
          walk_smem + (threadIdx.x >> 5) * fused_vecs<S, VA, TS>());
}

using FusedKernel = void (*)(const void *, void *, int, int, size_t, FusedStrips, long long, int, Coef, int,
                             const uint32_t *, uint32_t, const float *);

struct Choice {
    FusedKernel fn = nullptr;
    int smem = 0;
};

template <int S, int RND, int VA, int TS>
Choice choice() {
    return Choice{k_step_fused<S, RND, VA, TS>, kWarps * fused_vecs<S, VA, TS>() * 16};
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
    if (nx % fused_vec(storage) || (rnd && field)) return cudaSuccess;
    double best = 1e30;
    for (int steps = 2; steps <= fused_most_steps(storage); ++steps) {
        const Choice ch = choose(storage, rnd, field, steps);
        Err e = cudaFuncSetAttribute((const void *)ch.fn,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, ch.smem);
        if (e != cudaSuccess) return e;
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
    // Short tiles repeat too much of the earlier steps' work, and a launch of them
    // lasts one walk of eight rows or more however small the grid: single steps are
    // the faster where the tiles come out shorter than this.  Measured per step,
    // single steps against passes (rows in brackets): FP32 768^2 7.16 / 7.15 us (5),
    // 1024^2 10.97 / 9.41 (8), 2048^2 49.6 / 26.3 (32); with a c2 field 768^2 6.94 /
    // 7.51, 1024^2 11.75 / 9.89; FP16 1024^2 8.85 / 10.41 (5), 1536^2 15.22 / 15.02
    // (9), 2048^2 25.31 / 23.43 (16); with stochastic rounding, whose conversion is
    // the slower for FP16, BF16 1536^2 16.9 / 15.9 (9), 2048^2 27.6 / 24.9 (16), FP16
    // 2048^2 26.7 / 27.1 (16), 2048 x 4096 55.1 / 47.4 (31).
    const int least_rows = storage == ST_F32 ? 8 : (rnd && storage == ST_F16 ? 20 : 9);
    out->ok = out->rows >= least_rows;
    return cudaSuccess;
}

Err launch_fused(const FusedPlan &p, int storage, const void *fin, void *fout, int nx, int ny,
                 size_t P, const Coef &c, int steps, int rnd, const uint32_t *tdev, uint32_t toff,
                 const float *a15f, cudaStream_t st) {
    if (!p.ok) return cudaErrorInvalidValue;
    const Choice ch = choose(storage, rnd, a15f != nullptr, p.steps);
    return launch_pdl(ch.fn, (unsigned)((p.ntiles + kWarps - 1) / kWarps), 32u * kWarps,
                      (size_t)ch.smem, st, fin, fout, nx, ny, P, p.strips, p.ntiles, p.rows, c,
                      steps, tdev, toff, a15f);
}

}  // namespace vss

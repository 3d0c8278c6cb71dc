// The single-grid step kernel that advances two time steps per launch (the
// fused walk of lbm_walk2.cuh), and the plan that sizes its tiles.
#include "lbm_internal.h"
#include "lbm_launch.cuh"
#include "lbm_walk2.cuh"

namespace vss {

namespace {

constexpr int kWarps = 4;  // warps per block

// Bound: HBM for FP32, instruction issue for the 16-bit kinds (the fused walk
// halves the bytes per update).  Eight warps per SM of up to 255 registers, with
// two rows of copies in flight each: twelve warps at 168 registers, with the
// waiting row of step 1 in shared memory too, spent the time on shared-memory
// traffic in FP32 (71 % of its bandwidth; 8192^2 158k against 172k MLUPS) and
// spilled in the 16-bit kinds (214k against 245k).  Measured on one grid, per
// step, single steps before and pairs now: 8192^2 FP32 705.7 -> 392.4 us
// (171k MLUPS, 6.2 TB/s of the 36 B an update that two steps per pass need),
// FP16 372.5 -> 274.2 us (245k), BF16 with stochastic rounding 371.0 -> 296.5;
// 2048^2 49.6 -> 29.3, 25.3 -> 23.4; 2048^2 FP32 with a c2 field 54.0 -> 31.5.
template <int S, int RND, int VA>
__global__ void __launch_bounds__(32 * kWarps, 2)
    k_step2(const void *__restrict__ fin, void *__restrict__ fout, int nx, int ny, size_t P,
            int nstrips, long long ntiles, int rows, Coef c, const uint32_t *tdev, uint32_t toff,
            const float *__restrict__ a15f) {
    extern __shared__ uint4 walk_smem[];
    pdl_enter();
    const long long tile = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (tile >= ntiles) return;  // whole warps leave together
    const int strip = (int)(tile % nstrips), seg = (int)(tile / nstrips);
    const int y0 = seg * rows;
    Walker2<S, LD_NC, RND, VA> w(fin, fout, nx, ny, P, strip * Walk2Geom<S>::COLS);
    if constexpr (VA) w.a15f = a15f;
    if constexpr (RND) w.set_step((tdev ? *tdev : 0u) + toff);
    // Neighbouring segments walk in opposite directions, so the rows they
    // share are read by both at about the same time.
    w.run(y0, min(ny, y0 + rows), (seg & 1) ? -1 : 1, true, c,
          walk_smem + (threadIdx.x >> 5) * walk2_vecs<S, VA>());
}

using Step2Kernel = void (*)(const void *, void *, int, int, size_t, int, long long, int, Coef,
                             const uint32_t *, uint32_t, const float *);

struct Choice {
    Step2Kernel fn = nullptr;
    int smem = 0;
};

template <int S, int RND, int VA>
Choice choice() {
    return Choice{k_step2<S, RND, VA>, kWarps * walk2_vecs<S, VA>() * 16};
}

Choice choose(int storage, int rnd, bool field) {
    switch (storage) {
        case ST_F32:
            return field ? choice<ST_F32, 0, 1>() : choice<ST_F32, 0, 0>();
        case ST_F16:
            return field ? choice<ST_F16, 0, 1>()
                         : (rnd ? choice<ST_F16, 1, 0>() : choice<ST_F16, 0, 0>());
        case ST_BF16:
            return field ? choice<ST_BF16, 0, 1>()
                         : (rnd ? choice<ST_BF16, 1, 0>() : choice<ST_BF16, 0, 0>());
        default:
            return Choice{};
    }
}

}  // namespace

Err plan_step2(int storage, int rnd, bool field, int nx, int ny, Step2Plan *out) {
    *out = Step2Plan{};
    const int v = storage == ST_F32 ? 4 : 8;
    if (nx % v || (rnd && field)) return cudaSuccess;
    const Choice ch = choose(storage, rnd, field);
    Err e = cudaFuncSetAttribute((const void *)ch.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 ch.smem);
    if (e != cudaSuccess) return e;
    const long long wave = resident_warps((const void *)ch.fn, kWarps, ch.smem);
    if (wave <= 0) return cudaErrorLaunchOutOfResources;
    const int nstrips = (nx + 30 * v - 1) / (30 * v);
    // Tile height: a tile of r rows costs about r + 5 row steps (two rows of
    // the first step's collision and three pulled rows at each end), and a
    // launch lasts as many tiles as its fullest warp slot runs.  FP32 passes
    // are bound by HBM and run faster while the tiles in flight lie close
    // together, so their tiles stay within 64 rows.
    long long best = -1;
    int rows = 2;
    const int most = storage == ST_F32 ? 64 : 512;
    for (int r = 2; r <= most; ++r) {
        const long long tiles = (long long)nstrips * ((ny + r - 1) / r);
        const long long cost = ((tiles + wave - 1) / wave) * (r + 5);
        if (best < 0 || cost < best) {
            best = cost;
            rows = r;
        }
        if (r >= ny) break;
    }
    // Short tiles repeat too much of the first step's work, and a launch of them
    // lasts one walk of eight rows or more however small the grid: single steps
    // are the faster where the tiles come out shorter than this.  Measured per
    // step, single against pairs (rows in brackets): FP32 768^2 7.16 / 7.15 us
    // (5), 1024^2 10.97 / 9.41 (8), 2048^2 49.6 / 29.3 (31); FP32 with a c2
    // field 768^2 6.94 / 7.51, 1024^2 11.75 / 9.89; FP16 1024^2 8.85 / 10.41
    // (5), 1536^2 15.22 / 15.02 (9), 2048^2 25.31 / 23.43 (16); FP16 with
    // stochastic rounding 2048^2 26.7 / 27.1 (16), 2048 x 4096 55.1 / 47.4 (31).
    const int least = storage == ST_F32 ? 8 : (rnd ? 20 : 9);
    out->ok = rows >= least;
    out->rows = rows;
    out->nstrips = nstrips;
    out->ntiles = (long long)nstrips * ((ny + rows - 1) / rows);
    return cudaSuccess;
}

Err launch_step2(const Step2Plan &p, int storage, const void *fin, void *fout, int nx, int ny,
                 size_t P, const Coef &c, int rnd, const uint32_t *tdev, uint32_t toff,
                 const float *a15f, cudaStream_t st) {
    if (!p.ok) return cudaErrorInvalidValue;
    const Choice ch = choose(storage, rnd, a15f != nullptr);
    return launch_pdl(ch.fn, (unsigned)((p.ntiles + kWarps - 1) / kWarps), 32u * kWarps,
                      (size_t)ch.smem, st, fin, fout, nx, ny, P, p.nstrips, p.ntiles, p.rows, c,
                      tdev, toff, a15f);
}

}  // namespace vss

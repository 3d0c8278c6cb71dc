// Host side of the resident kernel (lbm_resident.cuh): the tiling of a grid and
// its launch.
#include <algorithm>

#include "lbm_internal.h"

namespace vss {

namespace {

struct Shape {
    int threads, rows;
};
// Block shapes: at most `threads` threads of `rows` rows each, as many rows as their
// registers hold: no kernel spills but FP32 768 x 3 without and 384 x 10 with a field (4
// and 20 bytes), FP16 384 x 10 with a field (16) and BF16 384 x 10 (4 to 44).  The order
// is that of the kernels (resident_of).
constexpr Shape kShapes[] = {{512, 1}, {512, 2}, {768, 2}, {768, 3}, {640, 4}, {512, 6}, {384, 10}};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);

// Threads and row pitch of an extended tile of W columns with K rows a thread:
// thread t has column t % Wt of band t / Wt.  K * pitch is Wt modulo 32, so the
// 32 lanes of a warp touch 32 banks also where they span several bands; Wt is
// W rounded up to what that needs (an idle column or three).
inline int lanes_for(int W, int K) {
    const int g = K & -K;  // the power of two in K
    return (W + g - 1) / g * g;
}
inline int pitch_for(int W, int K) {
    const int Wt = lanes_for(W, K);
    int p = W;
    while ((K * p - Wt) & 31) ++p;
    return p;
}

bool fits(int k, int W, int H) {
    const Shape s = kShapes[k];
    const int Wt = lanes_for(W, s.rows);
    return Wt <= s.threads && (s.threads / Wt) * s.rows >= H &&
           pitch_for(W, s.rows) * H <= s.threads * s.rows;
}

// Threads of a block, in whole warps.
int threads_for(int shape, int W, int H) {
    const int bands = (H + kShapes[shape].rows - 1) / kShapes[shape].rows;
    return (lanes_for(W, kShapes[shape].rows) * bands + 31) / 32 * 32;
}

int smem_of(int shape) { return 10 * kShapes[shape].threads * kShapes[shape].rows * 4; }

}  // namespace

// Time of a step in microseconds, fitted to measured launches of grids from 400 x 4
// to 600^2: two block barriers and the chain of a site's arithmetic, the warps'
// rows, and an exchange (two passes through L2 and the wait) shared by T steps.  An
// exchange of tiles whose edges lie on 32-byte sectors takes a fifth less (256^2 in
// 16 x 8 tiles 1.70 us a step, in 11 x 13 1.95; 8192 x 4 in 128 tiles 0.44, in 152
// 0.48).  Within a cluster it costs less for the few sites of a channel's tiles (400
// x 4: 0.44 -> 0.32 us a step) and no less for tiles cut in both directions (64^2:
// 1.06 against 1.07).
static double exchange_us(long long halo, bool aligned, bool cluster) {
    if (cluster) return 0.65 + 0.003 * (double)halo;
    return (2.4 + 0.0012 * (double)halo) * (aligned ? 0.8 : 1.0);
}
static double step_us(int shape, int W, int H, int hx, int hy, int T, bool aligned, bool cluster) {
    const double warp_rows = threads_for(shape, W, H) / 32 * kShapes[shape].rows;
    const int halo = W * H - (W - 2 * hx) * (H - 2 * hy);
    return 0.16 + 0.018 * warp_rows + (hx || hy ? exchange_us(halo, aligned, cluster) / T : 0.0);
}

constexpr int kClusterTiles = 16;  // the largest cluster (beyond the portable 8)

// The tiling with the lowest estimate.  Grids of up to about 660^2 sites have one.
bool may_run_resident(int nx, int ny, int sms) { return (long long)nx * ny <= 3900LL * sms; }

Err plan_resident(int nx, int ny, int sms, bool clusters, ResidentPlan *out) {
    *out = ResidentPlan{};
    if (!may_run_resident(nx, ny, sms)) return cudaSuccess;
    double best = 1e30;
    // (many tiles first: a good tiling early lets the bound below skip most others)
    for (int tx = 1; tx <= sms && tx <= nx; ++tx)
        for (int ty = std::min(sms / tx, ny); ty >= 1; --ty) {
            if ((long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty) > 3900) break;
            for (int T : {1, 2, 3, 4, 6, 8, 12, 16}) {
                if (tx * ty == 1 && T > 1) break;
                const int hx = tx > 1 ? 2 * T : 0, hy = ty > 1 ? 2 * T : 0;
                // a tile's halo lies in its neighbours
                if ((tx > 1 && nx / tx < hx) || (ty > 1 && ny / ty < hy)) break;
                const int W = (nx + tx - 1) / tx + 2 * hx, H = (ny + ty - 1) / ty + 2 * hy;
                const long long sites = (long long)W * H;
                if (sites > 3900) break;
                const int own = (W - 2 * hx) * (H - 2 * hy);
                const bool cluster = clusters && tx * ty > 1 && tx * ty <= kClusterTiles;
                const bool aligned = nx % tx == 0 && nx / tx % 8 == 0;
                const double least = 0.16 + 0.018 * (double)sites / 32 +
                                     (hx || hy ? exchange_us(sites - own, aligned, cluster) / T : 0.0);
                if (least >= best) continue;  // no shape can be better
                bool any = false;
                for (int k = 0; k < kNumShapes; ++k) {
                    if (!fits(k, W, H)) continue;
                    any = true;
                    const double us = step_us(k, W, H, hx, hy, T, aligned, cluster);
                    if (us >= best) continue;
                    best = us;
                    out->tx = tx;
                    out->ty = ty;
                    out->T = tx * ty == 1 ? 1 << 20 : T;
                    out->cluster = cluster;
                    out->shape = k;
                    out->threads = threads_for(k, W, H);
                    out->lanes = lanes_for(W, kShapes[k].rows);
                    out->pitch = pitch_for(W, kShapes[k].rows);
                    out->us = us;
                }
                if (!any) break;
            }
        }
    out->ok = best < 1e30;
    return cudaSuccess;
}

// Where a resident call pays.  A call of n steps costs about n r + L, r the step time of
// its kind and L the launch, the first load and the last store; the step kernel n t, or
// more in short calls, whose launches are not replayed.  Fitted to 600 pairs of
// measurements (100 sizes from 16^2 to 661^2 and from 4 to 16384 wide, calls of 4 to 512
// steps, each kind): the choice is the slower by more than 3 % for one in 200 of them.  The
// step kernel's time scatters by a fifth with where a grid's buffers lie in L2 (FP16 400 x
// 400 4.1 us, 400 x 408 5.1).  Step kernel / resident, us a step, calls of 4 and of 512
// steps: FP32 512^2 7.0 / 6.2 and 6.6 / 3.7, 640^2 7.3 / 8.2 and 6.8 / 6.0; FP32 with a c2
// field 512^2 5.2 / 6.7 and 4.8 / 4.4, 640^2 6.2 / 8.9 and 5.8 / 6.7; FP16 400^2 4.4 /
// 4.7 and 4.1 / 2.9, 640^2 6.2 / 8.7 and 5.9 / 6.2; FP16 with stochastic rounding, which
// hashes every site here but every pair of sites there, 400^2 4.4 / 6.0 and 4.4 / 4.0.
//
// `streams`: streams with small grids in use.  Their step kernels overlap, and so do
// resident calls as long as their tiles find SMs of their own, which is two grids of 64^2,
// eleven of 400 x 4, and none of 128^2 and more.  Measured, us per step and grid, step
// kernel / resident: FP32 64^2 on 4 streams 0.97 / 0.56, on 8 0.54 / 0.56; 128^2 on 2
// 1.93 / 1.17, on 8 0.64 / 1.17; 256^2 on 2 2.9 / 1.8, on 4 1.5 / 1.8, on 16 0.72 / 1.84;
// 512^2 on 2 3.6 / 3.7, on 4 2.3 / 3.7; FP16 512^2 on 4 1.9 / 4.0.
bool resident_pays(const ResidentPlan &p, int storage, int rnd, bool field, bool drive,
                   long long sites, int sms, int streams, long long n) {
    struct Kind {
        double t, per_site, most;           // of the step kernel
        double per_row, per_band, exchange; // beyond the plan's estimate
    };
    constexpr Kind kF32{2.6, 13e-6, 7.0, 0, 0.064, 0.9}, kF32Field{3.2, 7e-6, 5.8, 0, 0.11, 1.2};
    constexpr Kind k16{3.0, 10e-6, 6.0, 0, 0.088, 1.0}, k16Field{2.8, 15e-6, 6.0, 0, 0.135, 1.45};
    constexpr Kind kHash{3.6, 9e-6, 6.4, 0.0096, 0.145, 1.55};
    const bool wide = storage == ST_F32;
    const Kind k = wide ? (field ? kF32Field : kF32) : rnd ? kHash : field ? k16Field : k16;
    const int tiles = p.tx * p.ty;
    const double warp_rows = p.threads / 32 * kShapes[p.shape].rows;
    double t = std::min(k.t + k.per_site * (double)sites, k.most);
    if (drive) t += 2.5;  // the boundary kernel of every step
    double r = p.us - 0.24 + k.per_row * warp_rows + k.per_band * kShapes[p.shape].rows +
               (tiles > 1 ? k.exchange / p.T : 0.0);
    double fixed = 1.5 + 0.055 * warp_rows;
    if (streams > 1) {
        t = std::max({1.1 * t / streams, 0.45, (wide ? 8.5e-6 : 7e-6) * (double)sites});
        const int together = std::min(streams, std::max(1, sms / tiles));
        r /= together;
        fixed /= together;
    }
    return (double)n * (t - r) >= fixed;
}

static ResidentKernel kernel_for(const ResidentPlan &p, int storage, int rnd, bool field) {
    return storage == ST_F32   ? resident_kernel_f32(rnd, field, p.shape)
           : storage == ST_F16 ? resident_kernel_f16(rnd, field, p.shape)
                               : resident_kernel_bf16(rnd, field, p.shape);
}

// Launch parameters of a plan (attr: room for the cluster's attribute), and the
// attributes of its kernel, which are set again on each call at little cost.
static Err prepare_resident(const ResidentPlan &p, ResidentKernel fn, cudaStream_t st,
                            cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr) {
    const int smem = smem_of(p.shape);
    Err e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)(p.tx * p.ty));
    cfg->blockDim = dim3((unsigned)p.threads);
    cfg->dynamicSmemBytes = (size_t)smem;
    cfg->stream = st;
    cfg->attrs = attr;
    if (p.cluster) {
        e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        attr->id = cudaLaunchAttributeClusterDimension;
        attr->val.clusterDim.x = (unsigned)(p.tx * p.ty);
        attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
        cfg->numAttrs = 1;
    } else if (p.tx * p.ty > 1) {
        attr->id = cudaLaunchAttributeCooperative;
        attr->val.cooperative = 1;
        cfg->numAttrs = 1;
    }
    return e;
}

bool cluster_fits(const ResidentPlan &p, int storage, int rnd, bool field) {
    const ResidentKernel fn = kernel_for(p, storage, rnd, field);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    int clusters = 0;
    const bool ok = prepare_resident(p, fn, nullptr, &cfg, &attr) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, (const void *)fn, &cfg) == cudaSuccess;
    if (!ok) cudaGetLastError();
    return ok && clusters > 0;
}

Err launch_resident(const ResidentPlan &p, int storage, int rnd, ResidentArgs a, cudaStream_t st) {
    a.tx = p.tx;
    a.ty = p.ty;
    a.T = p.T;
    a.lanes = p.lanes;
    a.pitch = p.pitch;
    a.cluster = p.cluster ? 1 : 0;
    const ResidentKernel fn = kernel_for(p, storage, rnd, a.a15f != nullptr);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    const Err e = prepare_resident(p, fn, st, &cfg, &attr);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&a};
    return cudaLaunchKernelExC(&cfg, (const void *)fn, args);
}

}  // namespace vss

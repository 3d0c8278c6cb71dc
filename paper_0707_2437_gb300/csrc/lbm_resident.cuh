// Small grids: all steps of a call in one launch, with the state in shared
// memory.
//
// A grid that fits the SMs' shared memory (40 bytes a site) is cut into
// rectangular tiles, one per block.  A block keeps its tile's nine planes and a
// plane of drho in FP32 (16-bit storage: values rounded by every step as a
// store rounds them) and steps them in place:
//   A  every thread pulls its sites' nine values from the planes, forms drho
//      and writes it to its plane;
//   B  after a block barrier it collides them, with the neighbours' drho, and
//      writes the nine values back (all pulls are done by then).
// A thread owns K rows of one column, so the pulled values wait in registers
// and most y neighbours are its own.
//
// Tiles exchange edges through the grid's own two buffers, or, up to 16 of them, as
// one cluster (below).  A tile is extended
// by a halo of 2 T columns or rows in each direction in which the grid is cut;
// T steps use two sites of it each (the pull and the central difference), so
// the blocks meet once in T steps: a block writes its outer ring, raises its
// counter, waits for its eight neighbours' counters and reads their rings.  The
// buffers alternate from one exchange to the next: a neighbour that still reads
// the one before has not raised its counter for this one, which a block waits
// for before it writes again.  In a direction in which the grid is not cut the
// tile wraps on itself.
//
// Blocks wait for one another, so launches of several tiles are cooperative (all
// blocks resident, or none), every wait is bounded by the clock (lbm_set_timeout_us,
// read every 256 polls, or at every one under a limit of less than a millisecond), and
// a wait that runs out sets the handle's status word, at which the others give up too.
// Cluster barriers have no limit: the hardware starts a cluster whole, and every block
// reaches every one of them.
//
// Up to 16 tiles launch as one cluster instead, which the hardware schedules as a
// whole: a block reads its halo out of its neighbours' shared memory, between two
// cluster barriers (all tiles have done their steps; all halos have been read), of
// which the second is waited for only before the next step writes.  That takes about
// 0.7 us for a few dozen sites where flags and two passes through L2 take 2.2.
//
// The arithmetic is the Walker's, operation by operation.
#pragma once

#include "lbm_internal.h"
#include "lbm_fused.cuh"

namespace vss {

namespace {

__device__ __forceinline__ int first_of(int n, int parts, int i) {
    return (int)((long long)n * i / parts);
}
__device__ __forceinline__ int wrapped(int a, int n) {
    a %= n;
    return a < 0 ? a + n : a;
}

template <int S>
__device__ __forceinline__ float load_h(const void *f, size_t idx) {
    return elem_to_f<S>(load_elem<S, LD_CG>(reinterpret_cast<const typename StoreT<S>::T *>(f) + idx));
}
template <int S>
__device__ __forceinline__ void store_h(void *f, size_t idx, float v) {
    if constexpr (S == ST_F32)
        reinterpret_cast<float *>(f)[idx] = v;
    else  // exact: v is a value of the storage type
        reinterpret_cast<unsigned short *>(f)[idx] = (unsigned short)pack1<S>(v);
}
// The value a store of `v` leaves behind.
template <int S>
__device__ __forceinline__ float stored(float v) {
    if constexpr (S == ST_F32)
        return v;
    else
        return elem_to_f<S>(pack1<S>(v));
}
template <int S>
__device__ __forceinline__ float stored_d(double v) {
    if constexpr (S == ST_F32)
        return (float)v;
    else if constexpr (S == ST_F16)
        return __half2float(__double2half(v));
    else
        return __bfloat162float(__double2bfloat16(v));
}

__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A word of block `rank`'s shared memory, at the address `local` has here.
__device__ __forceinline__ uint32_t peer_address(uint32_t local, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ float peer_load(uint32_t address) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(address) : "memory");
    return v;
}

constexpr int kDriveChunk = 128;  // boundary values computed ahead

// NT threads of K rows each: up to NT * K sites of extended tile.
//
// Bound: the barriers and dependent chains of a step (about 0.2 us for tiles of a
// few hundred sites), the exchange (2.4 us and more, shared by T steps), then
// instruction issue (about 100 instructions a site, the halo's included).  The K
// rows of a thread are independent, so they overlap; more rows than ten spill.
// Measured per step, launches of step kernels before and resident now: 400 x 4 FP32
// 3.5 -> 0.33 us, driven 8192 x 4 FP32 7.5 -> 0.60, 64^2 3.5 -> 1.09, 256^2 4.2 ->
// 1.86, 509 x 381 5.4 -> 3.2, 512^2 6.6 -> 3.5; 512^2 FP16 5.6 -> 3.7, with stochastic
// rounding 6.2 -> 5.0.
template <int S, int RND, int VA, int NT, int K>
__global__ void __launch_bounds__(NT, 1)
    k_resident(ResidentArgs a) {
    constexpr int PS = NT * K;  // plane stride
    extern __shared__ float planes[];
    float *F = planes, *D = planes + 9 * PS;
    __shared__ float drive_h[kDriveChunk];
    const int bx = blockIdx.x % a.tx, by = blockIdx.x / a.tx;
    const int hx = a.tx > 1 ? 2 * a.T : 0, hy = a.ty > 1 ? 2 * a.T : 0;
    const int x0 = first_of(a.nx, a.tx, bx), x1 = first_of(a.nx, a.tx, bx + 1);
    const int y0 = first_of(a.ny, a.ty, by), y1 = first_of(a.ny, a.ty, by + 1);
    const int W = x1 - x0 + 2 * hx, H = y1 - y0 + 2 * hy;  // extended tile
    // The thread's column and rows of the extended tile.
    // Column t % lanes of band t / lanes (lanes and pitch are those of the widest
    // tile, which the plan fits to the planes).  Threads and rows past the tile's
    // wrap around in it: they repeat another thread's work on the same values and
    // write the same results, which costs no conditions in the steps.
    const int Wp = a.pitch, band = (int)threadIdx.x / a.lanes;
    const int xt = (int)threadIdx.x % a.lanes, x = xt % W;
    const int yb = band * K % H;
    const int gx = wrapped(x0 - hx + x, a.nx);
    const int xl = x == 0 ? W - 1 : x - 1, xr = x + 1 >= W ? 0 : x + 1;
    // Rows the thread moves between the planes and the buffers.
    const int rows = xt < W && band * K < H ? min(K, H - yb) : 0;
    int row[K + 2];  // offsets of rows yb - 1 .. yb + K
#pragma unroll
    for (int j = 0; j < K + 2; ++j) row[j] = wrapped(yb + j - 1, H) * Wp;
    const bool edge_col = a.drive && (gx == 0 || gx >= a.nx - 2);
    const bool own_x = x >= hx && x < W - hx;
    // Grid row of the thread's row j (which wraps in the tile first).
    auto grow = [&](int j) {
        int y = yb + j;
        while (y >= H) y -= H;
        return wrapped(y0 - hy + y, a.ny);
    };
    const Coef c = a.c;

    // One site from a buffer (element g of its planes), nine loads in flight.
    auto load_site = [&](const void *src, size_t g, float (&v)[9]) {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = load_h<S>(src, (size_t)i * a.P + g);
    };
    auto put_site = [&](int l, const float (&v)[9]) {
#pragma unroll
        for (int i = 0; i < 9; ++i) F[i * PS + l] = v[i];
    };
    // Frames of a rectangle of the tile: site m of the bx columns and by rows next
    // to the edges of a w x h rectangle, the rows first.  (Quotients of small
    // integers by a reciprocal: exact.)
    struct Frame {
        int w, h, bx, by, rows, sites;
        float per_w, per_b;
        __device__ __forceinline__ Frame(int w_, int h_, int bx_, int by_)
            : w(w_), h(h_), bx(bx_), by(by_) {
            // Edges that meet: the whole rectangle, as rows.
            rows = (2 * bx >= w || 2 * by >= h) ? h : 2 * by;
            sites = rows * w + (h - rows) * 2 * bx;
            per_w = 1.0f / (float)w;
            per_b = bx ? 0.5f / (float)bx : 0.f;
        }
        __device__ __forceinline__ void at(int m, int &fx, int &fy) const {
            if (m < rows * w) {
                fy = (int)(((float)m + 0.5f) * per_w);
                fx = m - fy * w;
                if (fy >= by && rows < h) fy += h - 2 * by;
            } else {
                m -= rows * w;
                fy = (int)(((float)m + 0.5f) * per_b);
                fx = m - fy * 2 * bx;
                if (fx >= bx) fx += w - 2 * bx;
                fy += by;
            }
        }
    };
    // The tile's outer ring of own sites (the neighbours' halos) to a buffer, and
    // its halo from one, spread evenly over the threads.
    const Frame ring(x1 - x0, y1 - y0, hx, hy), halo(W, H, hx, hy);
    auto write_ring = [&](void *dst) {
        for (int m = threadIdx.x; m < ring.sites; m += blockDim.x) {
            int fx, fy;
            ring.at(m, fx, fy);
            const int l = (fy + hy) * Wp + fx + hx;
            const size_t g = (size_t)(y0 + fy) * a.nx + (x0 + fx);
#pragma unroll
            for (int i = 0; i < 9; ++i) store_h<S>(dst, (size_t)i * a.P + g, F[i * PS + l]);
        }
    };
    auto halo_site = [&](int m, int &l, size_t &g) {
        int fx, fy;
        halo.at(m, fx, fy);
        int cx = x0 - hx + fx, cy = y0 - hy + fy;  // (halos lie in the neighbours)
        cx = cx < 0 ? cx + a.nx : (cx >= a.nx ? cx - a.nx : cx);
        cy = cy < 0 ? cy + a.ny : (cy >= a.ny ? cy - a.ny : cy);
        l = fy * Wp + fx;
        g = (size_t)cy * a.nx + cx;
    };
    // The same site in the neighbour that owns it: its block, and the offset there.
    const int left_w = x0 - first_of(a.nx, a.tx, wrapped(bx - 1, a.tx)) +
                       (bx == 0 ? a.nx : 0);  // width of the tile on the left
    const int up_h = y0 - first_of(a.ny, a.ty, wrapped(by - 1, a.ty)) + (by == 0 ? a.ny : 0);
    auto peer_site = [&](int m, int &rank, int &l) {
        int fx, fy;
        halo.at(m, fx, fy);
        int nbx = bx, nby = by, px = fx, py = fy;
        if (fx < hx) {
            nbx = bx == 0 ? a.tx - 1 : bx - 1;
            px = fx + left_w;
        } else if (fx >= W - hx) {
            nbx = bx + 1 == a.tx ? 0 : bx + 1;
            px = fx - (W - 2 * hx);
        }
        if (fy < hy) {
            nby = by == 0 ? a.ty - 1 : by - 1;
            py = fy + up_h;
        } else if (fy >= H - hy) {
            nby = by + 1 == a.ty ? 0 : by + 1;
            py = fy - (H - 2 * hy);
        }
        rank = nby * a.tx + nbx;
        l = py * Wp + px;
    };
    auto fetch_from_peers = [&] {
        const uint32_t planes_at = smem_u32(F);
        for (int m = threadIdx.x; m < halo.sites; m += blockDim.x) {
            int rank, l, fx, fy;
            peer_site(m, rank, l);
            const uint32_t from = peer_address(planes_at, rank) + 4u * (uint32_t)l;
            float v[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i] = peer_load(from + 4u * (uint32_t)(i * PS));
            halo.at(m, fx, fy);
            put_site(fy * Wp + fx, v);
        }
    };
    bool peers_read = true;  // no cluster barrier is open
    auto fetch_halo = [&](const void *src) {
        for (int m = threadIdx.x; m < halo.sites; m += 2 * blockDim.x) {
            const bool two = m + (int)blockDim.x < halo.sites;
            int l0, l1 = 0;
            size_t g0, g1 = 0;
            float v0[9], v1[9];
            halo_site(m, l0, g0);
            if (two) halo_site(m + blockDim.x, l1, g1);
            load_site(src, g0, v0);
            if (two) load_site(src, g1, v1);
            put_site(l0, v0);
            if (two) put_site(l1, v1);
        }
    };
    for (int j = 0; j < rows; j += 2) {
        float v0[9], v1[9];
        load_site(a.buf[a.cur], (size_t)grow(j) * a.nx + gx, v0);
        if (j + 1 < rows) load_site(a.buf[a.cur], (size_t)grow(j + 1) * a.nx + gx, v1);
        put_site((yb + j) * Wp + x, v0);
        if (j + 1 < rows) put_site((yb + j + 1) * Wp + x, v1);
    }
    __syncthreads();

    int out = a.cur ^ 1;  // the buffer of the next exchange, or of the result
    unsigned epoch = a.epoch;
    long long done = 0;
    bool ok = true;
    while (true) {
        const int steps = (int)min((long long)a.T, a.steps - done);
        for (int s = 0; s < steps; ++s) {
            const uint32_t t = a.t0 + (uint32_t)(done + s);
            if (a.drive) {
                const int at = (int)((done + s) % kDriveChunk);
                if (at == 0) {
                    // (the values of earlier steps have been used: barrier below)
                    for (int m = threadIdx.x; m < kDriveChunk; m += (int)blockDim.x)
                        drive_h[m] = stored_d<S>(
                            (1.0 + a.drive_amp * sin(6.283185307179586476925287 *
                                                     (double)(t + (uint32_t)m) / a.drive_period)) -
                            a.rho0);
                }
            }
            // The sites whose values are right shrink by two a step from the cut
            // edges; the others are computed all the same (in bounds, wrapped
            // in the tile) and not used, so that the K rows of a thread are one
            // straight run of code.
            //
            // A: pulls and drho.
            float h[K][9], dr[K], a15[K];
#pragma unroll
            for (int j = 0; j < K; ++j) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const int cx = EXi(i) > 0 ? xl : (EXi(i) < 0 ? xr : x);
                    h[j][i] = F[i * PS + row[j + 1 - EYi(i)] + cx];
                }
                a15[j] = VA ? __ldg(a.a15f + (size_t)grow(j) * a.nx + gx) : c.a15;
            }
#pragma unroll
            for (int j = 0; j < K; ++j) {
                dr[j] = delta_rho(h[j][0], h[j][1], h[j][2], h[j][3], h[j][4], h[j][5], h[j][6],
                                  h[j][7], h[j][8]);
                D[row[j + 1] + x] = dr[j];
            }
            __syncthreads();
            // B: collisions.
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const float dxm = D[row[j + 1] + xl], dxp = D[row[j + 1] + xr];
                const float dym = j > 0 ? dr[j > 0 ? j - 1 : 0] : D[row[0] + x];
                const float dyp = j + 1 < K ? dr[j + 1 < K ? j + 1 : j] : D[row[K + 1] + x];
                collide1(h[j], dr[j], __fsub_rn(dxp, dxm), __fsub_rn(dyp, dym), c, a15[j]);
                if constexpr (RND) {
                    const uint32_t site = (uint32_t)grow(j) * (uint32_t)a.nx + (uint32_t)gx;
                    const uint32_t base = sr_pair_base(site, sr_step_key(t));
                    const uint32_t sh = (site & 1u) * 16u;
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        h[j][i] = elem_to_f<S>(sr_round<S>(h[j][i], sr_word(base, i) >> sh));
                } else if constexpr (S != ST_F32) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) h[j][i] = stored<S>(h[j][i]);
                }
            }
            if (!peers_read) {  // (a cluster's first step after an exchange)
                cluster_wait();
                peers_read = true;
            }
            if (edge_col) {
                const float b = gx == 0 ? drive_h[(int)((done + s) % kDriveChunk)]
                                        : stored_d<S>(1.0 - a.rho0);
#pragma unroll
                for (int j = 0; j < K; ++j)
#pragma unroll
                    for (int i = 0; i < 9; ++i) h[j][i] = b;
            }
#pragma unroll
            for (int j = 0; j < K; ++j)
#pragma unroll
                for (int i = 0; i < 9; ++i) F[i * PS + row[j + 1] + x] = h[j][i];
            __syncthreads();
        }
        done += steps;
        if (done >= a.steps) break;
        if (a.cluster) {
            cluster_arrive();
            cluster_wait();
            fetch_from_peers();
            cluster_arrive();
            peers_read = false;
            __syncthreads();
            continue;
        }
        // Exchange: the outer ring of the tile's own sites out ...
        write_ring(a.buf[out]);
        ++epoch;
        if (a.tx * a.ty > 1) {
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.flags + 32 * blockIdx.x),
                             "r"(epoch)
                             : "memory");
            }
            // ... and the neighbours' rings in.
            if (threadIdx.x < 9) {
                const int nb = wrapped(by + (int)threadIdx.x / 3 - 1, a.ty) * a.tx +
                               wrapped(bx + (int)threadIdx.x % 3 - 1, a.tx);
                const unsigned *flag = a.flags + 32 * nb;
                unsigned long long began = 0;
                for (unsigned it = 0;; ++it) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                                 : "=r"(v)
                                 : "l"(flag)
                                 : "memory");
                    if ((int)(v - epoch) >= 0) break;
                    if ((it & a.wait_polls) == a.wait_polls) {
                        const unsigned long long now = globaltimer_ns();
                        if (began == 0) began = now;
                        if (now - began >= a.wait_ns || *(volatile int *)a.status != 0) {
                            atomicCAS(a.status, 0, STATUS_TIMEOUT);
                            ok = false;
                            break;
                        }
                    }
                }
            }
            if (__syncthreads_or(!ok)) return;
            fetch_halo(a.buf[out]);
        }
        out ^= 1;
        __syncthreads();
    }
    for (int j = 0; j < rows; ++j) {
        if (!own_x || yb + j < hy || yb + j >= H - hy) continue;
        const size_t g = (size_t)grow(j) * a.nx + gx;
#pragma unroll
        for (int i = 0; i < 9; ++i)
            store_h<S>(a.buf[out], (size_t)i * a.P + g, F[i * PS + (yb + j) * Wp + x]);
    }
}

template <int S, int RND, int VA>
ResidentKernel resident_of(int shape) {
    switch (shape) {
        case 0:
            return k_resident<S, RND, VA, 512, 1>;
        case 1:
            return k_resident<S, RND, VA, 512, 2>;
        case 2:
            return k_resident<S, RND, VA, 768, 2>;
        case 3:
            return k_resident<S, RND, VA, 768, 3>;
        case 4:
            return k_resident<S, RND, VA, 640, 4>;
        case 5:
            return k_resident<S, RND, VA, 512, 6>;
        default:
            return k_resident<S, RND, VA, 384, 10>;
    }
}
}  // namespace

}  // namespace vss

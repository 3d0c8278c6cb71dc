// Several time steps per pass over memory: the fused strip walk.
//
// A pass of T steps reads buffer A and writes the state T steps later into buffer
// B; the states in between never leave the SM.  One warp owns a strip of columns
// (V = 16 bytes of elements per lane) and loads halo lanes on both sides.  A step
// reaches two columns (the pull, then the central difference of the pulled
// density), T steps reach 2 T, which the halo lanes' columns cover (one lane a
// side for T = 2, two for FP32's T = 3), so the strip needs no other halo work:
// every shuffle stays inside the warp, and what the outer lanes compute from their
// missing neighbours reaches no stored site.  Columns wrap lane by lane where nx is a
// multiple of V, and 4-byte word by word where it is not (RAG below).
//
// Down the rows the walk is a pipeline of T stages.  Each iteration takes a row of
// stored values, copied ahead into shared memory (cp.async), and for each stage
//   1. shifts it into the pulled row and forms its drho;
//   2. collides the row the stage pulled before, which gives that row after the
//      stage's step, rounded as a store would round it (the last stage stores it);
//   3. assembles the next stage's pulled row, one row behind, from this row and the
//      two before it.
// Two rows of copies are in flight.  The first stage's pulled row waits for its
// collision in registers; those of the later stages, and the six vectors of rows
// between two stages that a later row pulls, wait in shared memory, at the lane
// that wrote them.  A segment of n rows pulls n + 4 T - 2 rows; stage s = 0 .. T-1
// collides n + 4 (T - 1 - s).
//
// The arithmetic is the Walker's, operation by operation, so a pass leaves bit for
// bit the state that T single steps leave.
#pragma once

#include "lbm_internal.h"

namespace vss {

// x - y with one rounding, as a packed fused multiply-add (y * -1 is exact).
__device__ __forceinline__ float2 sub2(float2 x, float2 y) {
    return __ffma2_rn(y, make_float2(-1.f, -1.f), x);
}
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

// delta_rho of two sites.
__device__ __forceinline__ float2 delta_rho2(const float2 (&h)[9]) {
    const float2 sa = __fadd2_rn(__fadd2_rn(h[1], h[2]), __fadd2_rn(h[3], h[4]));
    const float2 sd = __fadd2_rn(__fadd2_rn(h[5], h[6]), __fadd2_rn(h[7], h[8]));
    return __ffma2_rn(both(VSS_W0), h[0],
                      __ffma2_rn(both(VSS_W1), sa, __fmul2_rn(both(VSS_W5), sd)));
}

// Collision of two sites in place: site_quantities and pair_out with packed
// operations.  gx, gy: drho differences across the sites; a15: alpha factors.
__device__ __forceinline__ void collide2(float2 (&h)[9], float2 dr, float2 gx, float2 gy,
                                         const Coef &c, float2 a15) {
    const float2 a = sub2(h[5], h[7]), b = sub2(h[6], h[8]);
    const float2 jx = __ffma2_rn(both(VSS_W1), sub2(h[1], h[3]),
                                 __fmul2_rn(both(VSS_W5), sub2(a, b)));
    const float2 jy = __ffma2_rn(both(VSS_W1), sub2(h[2], h[4]),
                                 __fmul2_rn(both(VSS_W5), __fadd2_rn(a, b)));
    const float2 rho = __fadd2_rn(both(c.rho0), dr);
    const float2 inv = make_float2(rcp_approx(rho.x), rcp_approx(rho.y));
    const float2 ux = __fmul2_rn(jx, inv), uy = __fmul2_rn(jy, inv);
    const float2 ju = __ffma2_rn(jx, ux, __fmul2_rn(jy, uy));
    const float2 wB = __fmul2_rn(both(c.om), __ffma2_rn(both(-1.5f), ju, dr));
    const float2 Ax = __ffma2_rn(both(c.w3), jx,
                                 __ffma2_rn(both(c.w3lo), jx, __fmul2_rn(a15, gx)));
    const float2 Ay = __ffma2_rn(both(c.w3), jy,
                                 __ffma2_rn(both(c.w3lo), jy, __fmul2_rn(a15, gy)));
    h[0] = __ffma2_rn(both(c.om1), h[0], wB);
    auto pair = [&](float2 &hi, float2 &ho, float2 ej, float2 eu, float2 eA) {
        const float2 s = __ffma2_rn(both(c.w45), __fmul2_rn(ej, eu), wB);
        hi = __fadd2_rn(__ffma2_rn(both(c.om1), hi, s), eA);
        ho = sub2(__ffma2_rn(both(c.om1), ho, s), eA);
    };
    pair(h[1], h[3], jx, ux, Ax);
    pair(h[2], h[4], jy, uy, Ay);
    pair(h[5], h[7], __fadd2_rn(jx, jy), __fadd2_rn(ux, uy), __fadd2_rn(Ax, Ay));
    pair(h[6], h[8], sub2(jy, jx), sub2(uy, ux), sub2(Ay, Ax));
}

// The same for one site.
__device__ __forceinline__ void collide1(float (&h)[9], float dr, float gx, float gy,
                                         const Coef &c, float a15) {
    const SiteQ q = site_quantities(h[1], h[2], h[3], h[4], h[5], h[6], h[7], h[8], dr, gx, gy,
                                    c, a15);
    float o[9];
    o[0] = __fmaf_rn(c.om1, h[0], q.wB);
    pair_out(h[1], h[3], q.jx, q.ux, q.Ax, q.wB, c, o[1], o[3]);
    pair_out(h[2], h[4], q.jy, q.uy, q.Ay, q.wB, c, o[2], o[4]);
    pair_out(h[5], h[7], __fadd_rn(q.jx, q.jy), __fadd_rn(q.ux, q.uy), __fadd_rn(q.Ax, q.Ay),
             q.wB, c, o[5], o[7]);
    pair_out(h[6], h[8], __fsub_rn(q.jy, q.jx), __fsub_rn(q.uy, q.ux), __fsub_rn(q.Ay, q.Ax),
             q.wB, c, o[6], o[8]);
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = o[i];
}

// A walk of TS steps.  The 16-bit kinds take two steps a pass, which leaves them bound
// by instruction issue.  FP32 takes two or three: at two it is bound by HBM and wants
// tiles close together, at three by shared memory and issue, with more rows and
// columns of halo, so it pays where tiles are tall (8192^2 174k against 203k MLUPS,
// 1024^2 112k against 105k; four steps leave shared memory for six warps per SM and
// run at 160k). 
template <int S, int TS>
struct FusedGeom {
    static constexpr int V = (S == ST_F32) ? 4 : 8;     // sites per lane, 16 bytes
    static constexpr int HALO = (2 * TS + V - 1) / V;   // halo lanes a side
    static constexpr int COLS = (32 - 2 * HALO) * V;    // columns a strip stores
};
// A width of a whole number of words of 4 bytes, of at least a lane's vector.
inline bool fused_width(int storage, int nx) {
    return storage == ST_F32 ? nx >= 4 : nx >= 8 && nx % 2 == 0;
}
constexpr int fused_vec(int storage) { return storage == ST_F32 ? 4 : 8; }
constexpr int fused_cols(int storage, int steps) {
    return storage == ST_F32 ? (steps == 3 ? FusedGeom<ST_F32, 3>::COLS : FusedGeom<ST_F32, 2>::COLS)
                             : FusedGeom<ST_F16, 2>::COLS;
}
constexpr int fused_most_steps(int storage) { return storage == ST_F32 ? 3 : 2; }
// Tallest tiles: FP32's passes of two steps are bound by HBM and run faster while the
// tiles in flight lie close together (8192^2, 48 rows 385 us a step, 235 rows 419).
constexpr int fused_most_rows(int storage, int steps) {
    return storage == ST_F32 && steps == 2 ? 64 : 512;
}

// The strips of nx columns (a multiple of fused_vec where tiles are packed).  Packing
// saves walks of mostly idle lanes, which pays in the 16-bit kinds, bound by issue: FP16
// 4096^2 76.2 -> 71.8
// us a step, 8192^2 279 -> 272, 512 uneven FP16 grids in a batch 209k -> 229k MLUPS.
// FP32 passes are bound by memory and gain nothing (2048^2 with three steps 26.3 /
// 26.4 us; 512 uneven grids 178k / 174k), and as the lanes of a packed tile read and
// write far apart it walks more slowly than the others (2048^2 with a c2 field and two
// steps 31.2 / 39.9 us, eight pieces).
constexpr bool fused_packs(int storage) { return storage != ST_F32; }
inline FusedStrips fused_strips(int storage, int steps, int nx) {
    const int vec = fused_vec(storage), use = fused_cols(storage, steps) / vec, halo = 32 - use;
    const int n = (nx + vec - 1) / vec, rest = n % use, pieces = rest ? 32 / (rest + halo) : 0;
    if (pieces == 1 || (rest && (!fused_packs(storage) || nx % vec))) return {n / use + 1, 0, 0};
    return {n / use, rest + halo, pieces};
}
// Row steps a tile costs beyond its rows (the pulls and collisions at its ends).
constexpr int fused_overhead(int steps) { return 4 * steps - 3; }

// Shared memory of one warp, in 16-byte vectors: two landing rows; for each stage
// after the first the rows held for it and the row that waits in it; with a c2
// field the alpha values of the rows in flight.
// FP32 with a c2 field takes all of it for three stages; the alpha values of the rows
// in flight then move down five vectors of registers, one per iteration (2048^2
// 31.2 -> 29.9 us a step against two stages, 4096^2 114.3 -> 102.4; each stage loading
// its own row an iteration ahead took 30.4 and 104.7).
template <int S, int TS>
constexpr bool fused_alpha_ring() {
    return S != ST_F32 || TS < 3;
}
// RAG: a staging row for the stores.
template <int S, int VA, int TS, bool RAG = false>
constexpr int fused_vecs() {
    return (2 + 2 * (TS - 1) + (RAG ? 1 : 0)) * 9 * 32 +
           (VA && fused_alpha_ring<S, TS>() ? (2 * TS + 2) * (FusedGeom<S, TS>::V / 4) * 32 : 0);
}

// PACK: tiles may be packed.  Otherwise the rows are the warp's, not the lane's, which
// saves about 1 % (nine FP32 grids of 2048^2 in the flow schedule 173.6k / 174.4k).
// RAG: a width that is no multiple of the lanes' vectors.  Rows then start at any word
// of 4 bytes, so they are copied word by word, lane after lane along the row (the
// shared-memory image of a row is the same), and stored that way from a staging row.
template <int S, int LD, int RND, int VA, int TS, bool PACK, bool RAG = false>
struct FusedWalk {
    static_assert(!RAG || (LD == LD_NC && !VA && !PACK),
                  "4-byte copies go through L1; no alpha rows, whole strips");
    static constexpr int WS = FusedGeom<S, TS>::V / 4;  // sites of a word
    int col[RAG ? 4 : 1] = {};  // RAG: the column of words lane, lane + 32, ... of a row,
    uint32_t mine = 0;          // and the ones among them that the strip stores
    static constexpr int V = FusedGeom<S, TS>::V;
    static constexpr int HALO = FusedGeom<S, TS>::HALO;
    static_assert(Pack<S, V>::NW == 4, "a lane holds one 16-byte vector per direction");
    static_assert(RND == 0 || S != ST_F32, "stochastic rounding applies to 16-bit storage");
    using T = typename StoreT<S>::T;
    static constexpr int AV = V / 4;      // alpha vectors of a lane's sites
    static constexpr int AS = 2 * TS + 2;  // slots of alpha rows in shared memory
    static constexpr int AL = 2 * TS - 1;  // rows of them kept in registers instead
    static constexpr bool RING = VA && fused_alpha_ring<S, TS>();
    uint32_t rkey[TS] = {};  // sr_step_key of the steps
    const float *__restrict__ a15f = nullptr;

    const T *__restrict__ fin;
    T *__restrict__ fout;
    int nx, ny;
    size_t P;
    int lane, xl;
    int ylo, own;  // the lane's rows: own of them from ylo (0: none)

    // Columns from x0 and rows y0 .. y1-1, cut into pieces of `rows` rows (y1 - y0: one)
    // on `lanes` lanes each (32: one).
    __device__ __forceinline__ FusedWalk(const void *fin_, void *fout_, int nx_, int ny_, size_t P_,
                                         int x0, int y0, int y1, int rows, int lanes)
        : fin(reinterpret_cast<const T *>(fin_)),
          fout(reinterpret_cast<T *>(fout_)),
          nx(nx_),
          ny(ny_),
          P(P_) {
        lane = threadIdx.x & 31;
        const int piece = PACK ? lane / lanes : 0, at = lane - piece * lanes;
        const int xu = x0 + (at - HALO) * V;  // the lane's columns, unwrapped
        ylo = y0 + piece * rows;
        const bool act = at >= HALO && at < lanes - HALO && xu < nx && (piece + 1) * lanes <= 32;
        own = act ? (PACK ? max(0, min(rows, y1 - ylo)) : rows) : 0;
        xl = xu % nx;
        if (xl < 0) xl += nx;
        if constexpr (RAG) {
            own = rows;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int w = 32 * j + lane, x = x0 + (w - 4 * HALO) * WS;
                if (w >= 4 * HALO && w < 4 * (32 - HALO) && x < nx) mine |= 1u << j;
                col[j] = x % nx;
                if (col[j] < 0) col[j] += nx;
            }
        }
    }
    __device__ __forceinline__ void set_step(uint32_t step) {
#pragma unroll
        for (int s = 0; s < TS; ++s) rkey[s] = sr_step_key(step + (uint32_t)s);
    }

    __device__ __forceinline__ static void take(uint32_t (&w)[9][4], const uint4 *s) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const uint4 u = s[i * 32];
            w[i][0] = u.x;
            w[i][1] = u.y;
            w[i][2] = u.z;
            w[i][3] = u.w;
        }
    }
    __device__ __forceinline__ static void keep(uint4 *s, const uint32_t (&w)[9][4]) {
#pragma unroll
        for (int i = 0; i < 9; ++i) s[i * 32] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
    }

    // Copies the lane's nine vectors of pulled row q0 (and its alpha values)
    // into shared memory, as one commit group.
    __device__ __forceinline__ void issue(int qm, int q0, int qp, uint4 *land, uint4 *al) const {
        if constexpr (RAG) {
            __syncwarp();  // the row before has been taken by every lane
            const uint32_t to = (uint32_t)__cvta_generic_to_shared(land - lane) + 4 * lane;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int sr = (EYi(i) > 0) ? qm : ((EYi(i) < 0) ? qp : q0);
                const T *src = fin + ((size_t)i * P + (size_t)sr * nx);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                     to + 512 * i + 128 * j),
                                 "l"(src + col[j])
                                 : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            return;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int sr = (EYi(i) > 0) ? qm : ((EYi(i) < 0) ? qp : q0);
            const T *src = fin + ((size_t)i * P + (size_t)sr * nx + xl);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(land + i * 32)),
                         "l"(src)
                         : "memory");
        }
        if constexpr (RING) {
#pragma unroll
            for (int h = 0; h < AV; ++h)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(al + h * 32)),
                             "l"(a15f + (size_t)q0 * nx + xl + 4 * h)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }

    // Shifts of the e_x = +-1 directions and drho of the lane's sites.
    __device__ __forceinline__ void finish(uint32_t (&w)[9][4], float (&d)[V]) const {
        shift_from_left<S, V>(w[1], __shfl_up_sync(FULL, w[1][3], 1));
        shift_from_left<S, V>(w[5], __shfl_up_sync(FULL, w[5][3], 1));
        shift_from_left<S, V>(w[8], __shfl_up_sync(FULL, w[8][3], 1));
        shift_from_right<S, V>(w[3], __shfl_down_sync(FULL, w[3][0], 1));
        shift_from_right<S, V>(w[6], __shfl_down_sync(FULL, w[6][0], 1));
        shift_from_right<S, V>(w[7], __shfl_down_sync(FULL, w[7][0], 1));
        if constexpr (S == ST_F32) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float h[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = __uint_as_float(w[i][v]);
                d[v] = delta_rho(h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7], h[8]);
            }
        } else {
#pragma unroll
            for (int v = 0; v < V; v += 2) {
                float2 h[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = unpack2<S>(w[i][v >> 1]);
                const float2 r = delta_rho2(h);
                d[v] = r.x;
                d[v + 1] = r.y;
            }
        }
    }

    // Collides the pulled row r in place.  d: its drho; before, after: drho of
    // the rows walked before and after it; dir: the walking direction as +1 or
    // -1, a factor of the y difference (exact, and one code for both).
    __device__ __forceinline__ void collide(int r, uint32_t (&w)[9][4], const float (&d)[V],
                                            const float (&before)[V], const float (&after)[V],
                                            float dir, const Coef &c, uint32_t rkey,
                                            const uint4 (&al)[AV]) const {
        const float lft = __shfl_up_sync(FULL, d[V - 1], 1);
        const float rgt = __shfl_down_sync(FULL, d[0], 1);
        float a15v[V];
        if constexpr (VA) {
#pragma unroll
            for (int h = 0; h < V / 4; ++h) {
                const uint4 u = al[h];
                a15v[4 * h + 0] = __uint_as_float(u.x);
                a15v[4 * h + 1] = __uint_as_float(u.y);
                a15v[4 * h + 2] = __uint_as_float(u.z);
                a15v[4 * h + 3] = __uint_as_float(u.w);
            }
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) a15v[v] = c.a15;
        }
        if constexpr (S == ST_F32) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float h[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = __uint_as_float(w[i][v]);
                const float gx = __fsub_rn(v == V - 1 ? rgt : d[v + 1], v == 0 ? lft : d[v - 1]);
                const float gy = __fmaf_rn(dir, after[v], __fmul_rn(-dir, before[v]));
                collide1(h, d[v], gx, gy, c, a15v[v]);
#pragma unroll
                for (int i = 0; i < 9; ++i) w[i][v] = __float_as_uint(h[i]);
            }
        } else {
#pragma unroll
            for (int v = 0; v < V; v += 2) {
                float2 h[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = unpack2<S>(w[i][v >> 1]);
                const float2 gx = make_float2(__fsub_rn(d[v + 1], v == 0 ? lft : d[v - 1]),
                                              __fsub_rn(v + 2 == V ? rgt : d[v + 2], d[v]));
                const float2 gy =
                    __ffma2_rn(both(dir), make_float2(after[v], after[v + 1]),
                               __fmul2_rn(both(-dir), make_float2(before[v], before[v + 1])));
                collide2(h, make_float2(d[v], d[v + 1]), gx, gy, c,
                         make_float2(a15v[v], a15v[v + 1]));
                if constexpr (RND) {
                    // nx and v are even: the two sites are a hash pair
                    int x = xl + v;
                    if (RAG && x >= nx) x -= nx;
                    const uint32_t base =
                        sr_pair_base((uint32_t)r * (uint32_t)nx + (uint32_t)x, rkey);
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        w[i][v >> 1] = sr_pack2<S>(h[i].x, h[i].y, sr_word(base, i));
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i) w[i][v >> 1] = pack2<S>(h[i].x, h[i].y);
                }
            }
        }
    }

    __device__ __forceinline__ void store(int r, const uint32_t (&w)[9][4], uint4 *buf) const {
        if constexpr (RAG) {
            uint4 *stage = buf + (2 + 2 * (TS - 1)) * 9 * 32;
            keep(stage + lane, w);
            __syncwarp();
            const uint32_t *from = reinterpret_cast<const uint32_t *>(stage) + lane;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                T *dst = fout + ((size_t)i * P + (size_t)r * nx);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (mine >> j & 1)
                        *reinterpret_cast<uint32_t *>(dst + col[j]) = from[128 * i + 32 * j];
            }
            return;
        }
        if (PACK ? (unsigned)(r - ylo) >= (unsigned)own : own == 0) return;
        T *dst = fout + ((size_t)r * nx + xl);
#pragma unroll
        for (int i = 0; i < 9; ++i) store_words<S, V>(dst + (size_t)i * P, w[i]);
    }

    // For stage s >= 1: the held rows, [0..2] e_y = 0 of the last row, [3..5] and
    // [6..8] the late trio of the last two rows; the waiting row.  The alpha values.
    __device__ __forceinline__ uint4 *held_of(uint4 *buf, int s) const {
        return buf + (18 + 18 * (s - 1)) * 32 + lane;
    }
    __device__ __forceinline__ uint4 *wait_of(uint4 *buf, int s) const {
        return buf + (27 + 18 * (s - 1)) * 32 + lane;
    }
    __device__ __forceinline__ uint4 *alpha_of(uint4 *buf) const {
        return buf + (18 + 18 * (TS - 1)) * 32 + lane;
    }

    // Iteration k of stage SG and the stages after it.  The stage pulls from iteration
    // 4 SG on and collides from 4 SG + 2 on; u holds its waiting row.  d: drho per
    // stage of the rows pulled two, one and zero iterations ago; row: the pulled row
    // of the first stage, ia its alpha slot; back[s]: rows from it to stage s's.
    template <int SG>
    __device__ __forceinline__ void stage(int k, int dir, int steps, float sgn, const Coef &c,
                                          int ia, uint4 *buf, uint32_t (&u)[9][4],
                                          float (&d)[TS][3][V], int row, const int (&back)[TS],
                                          const uint4 (&alpha)[AL][AV]) const {
        if (k < 4 * SG + 2) return;
        int r = row - back[SG];
        if (r < 0) r += ny;
        if constexpr (RING) {
            const int as = ia - (2 * SG + 1);
            const uint4 *from = alpha_of(buf) + (as < 0 ? as + AS : as) * AV * 32;
            uint4 a[AV];
#pragma unroll
            for (int h = 0; h < AV; ++h) a[h] = from[h * 32];
            collide(r, u, d[SG][1], d[SG][0], d[SG][2], sgn, c, rkey[SG], a);
        } else {
            collide(r, u, d[SG][1], d[SG][0], d[SG][2], sgn, c, rkey[SG], alpha[2 * SG]);
        }
        if constexpr (SG + 1 < TS) {
            if (SG + 1 < steps) {
                // The row after this stage is in u.  The next stage's pulled row, one
                // behind, takes e_y = 0 from the row before and, in walking order, one
                // trio of an axis and two diagonals from this row and the other from
                // two rows before.
                uint4 *held = held_of(buf, SG + 1), *late = held + (3 + 3 * (k & 1)) * 32;
                auto swap = [&](int i, uint4 *place) {
                    const uint4 o = *place;
                    *place = make_uint4(u[i][0], u[i][1], u[i][2], u[i][3]);
                    u[i][0] = o.x;
                    u[i][1] = o.y;
                    u[i][2] = o.z;
                    u[i][3] = o.w;
                };
                swap(0, held);
                swap(1, held + 32);
                swap(3, held + 64);
                if (dir > 0) {
                    swap(2, late);
                    swap(5, late + 32);
                    swap(6, late + 64);
                } else {
                    swap(4, late);
                    swap(7, late + 32);
                    swap(8, late + 64);
                }
                if (k >= 4 * (SG + 1)) {
                    finish(u, d[SG + 1][2]);
                    // This row waits; the one that waited is collided next.
                    uint4 *wait = wait_of(buf, SG + 1);
                    if (k >= 4 * (SG + 1) + 2) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) swap(i, wait + i * 32);
                        stage<SG + 1>(k, dir, steps, sgn, c, ia, buf, u, d, row, back, alpha);
                    } else {
                        keep(wait, u);
                    }
                }
                return;
            }
        }
        store(r, u, buf);
    }

    // Advances the pieces' rows (`rows` each, not above ny; walked by all pieces, stored
    // where they are the lane's) by `steps` (1 .. TS) steps in direction dir.  `buf`:
    // the warp's fused_vecs() vectors.
    __device__ __forceinline__ void run(int rows, int dir, int steps, const Coef &c,
                                        uint4 *buf) const {
        uint4 *land = buf + lane;  // two slots
        uint4 *al = alpha_of(buf);
        const float sgn = dir > 0 ? 1.f : -1.f;
        const int ext = 2 * steps - 1;
        const int K = rows + 2 * ext;
        // The next row to copy (wrapped) and the rows before and after it.
        int q0 = (dir > 0 ? ylo - ext : ylo + rows - 1 + ext) % ny;
        if (q0 < 0) q0 += ny;
        int qm = (q0 == 0) ? ny - 1 : q0 - 1;
        int qp = (q0 + 1 == ny) ? 0 : q0 + 1;
        auto next = [&] {
            if (dir > 0) {
                qm = q0;
                q0 = qp;
                qp = (qp + 1 == ny) ? 0 : qp + 1;
            } else {
                qp = q0;
                q0 = qm;
                qm = (qm == 0) ? ny - 1 : qm - 1;
            }
        };
        int row = q0;  // the pulled row of the first stage
        int back[TS];  // stage s collides the row pulled 2 s + 1 iterations ago
#pragma unroll
        for (int j = 0; j < TS; ++j) {
            back[j] = (2 * j + 1) * dir % ny;
            if (back[j] < 0) back[j] += ny;
        }

        uint32_t wc[9][4] = {};  // the first stage's waiting row
        float d[TS][3][V];       // per stage: drho of the rows pulled two, one, zero ago
#pragma unroll
        for (int s = 0; s < TS; ++s)
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int v = 0; v < V; ++v) d[s][j][v] = 0.f;
        int ia = 0;  // alpha slot of the pulled row, mod AS
        uint4 alpha[AL][AV] = {};  // of the rows pulled one iteration ago, two, ...
        uint4 fresh = make_uint4(0, 0, 0, 0);
        issue(qm, q0, qp, land, al);
        next();
        issue(qm, q0, qp, land + 9 * 32, al + AV * 32);  // K >= 3
        next();
        for (int k = 0; k < K; ++k) {
            uint32_t w[9][4], u[9][4];
            uint4 *slot = land + (k & 1) * 9 * 32;
            if constexpr (VA && !RING)
                fresh = __ldg(reinterpret_cast<const uint4 *>(a15f + (size_t)row * nx + xl));
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            if constexpr (RAG) __syncwarp();  // the other lanes' copies too
            take(w, slot);
            finish(w, d[0][2]);
            // The words read from the landing row have been used (the
            // shuffles), so the next copy cannot overtake them.
            if (k + 2 < K) {
                issue(qm, q0, qp, slot, al + (ia < AS - 2 ? ia + 2 : ia + 2 - AS) * AV * 32);
                next();
            } else {
                asm volatile("cp.async.commit_group;" ::: "memory");  // keeps the count
            }
#pragma unroll
            for (int i = 0; i < 9; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    u[i][j] = wc[i][j];
                    wc[i][j] = w[i][j];
                }
            stage<0>(k, dir, steps, sgn, c, ia, buf, u, d, row, back, alpha);
#pragma unroll
            for (int s = 0; s < TS; ++s)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    d[s][0][v] = d[s][1][v];
                    d[s][1][v] = d[s][2][v];
                }
            row += dir;
            if (row < 0) row += ny;
            if (row >= ny) row -= ny;
            if constexpr (VA && !RING) {
#pragma unroll
                for (int j = AL - 1; j > 0; --j) alpha[j][0] = alpha[j - 1][0];
                alpha[0][0] = fresh;
            }
            ia = ia == AS - 1 ? 0 : ia + 1;
        }
    }
};

}  // namespace vss

// Two time steps per pass over memory: the fused strip walk.
//
// A pass reads buffer A and writes the state two steps later into buffer B;
// the state in between never leaves the SM.  One warp owns a strip of 30 V
// columns (V = 16 bytes of elements per lane) and loads 32 V: the two outer
// lanes hold halo columns.  A step reaches two columns (the pull, then the
// central difference of the pulled density), two steps reach four, and V is 4
// or 8, so the outer lanes' columns cover it and the strip needs no other halo
// work: every shuffle stays inside the warp, and what the outer lanes compute
// from their missing neighbours reaches no stored site.  Columns wrap lane by
// lane, so nx must be a multiple of V.
//
// Down the rows the walk is a pipeline of two stages.  Each iteration
//   1. takes a row of stored values, copied ahead into shared memory
//      (cp.async), shifts it into the pulled row p and forms its drho;
//   2. collides the row pulled before, which gives row q = p - 1 after step 1
//      (all "-1" in walking order), rounded as a store would round it;
//   3. assembles the pulled row s = q - 1 of step 2 from the rows q, q - 1 and
//      q - 2 after step 1 and forms its drho;
//   4. collides row s - 1, which gives the row after step 2, and stores it.
// Two rows of copies are in flight.  The pulled row of step 1 waits for its
// collision in registers, the one of step 2 and the six vectors of rows after
// step 1 that a later row pulls wait in shared memory, at the lane that wrote
// them.  A segment of n rows pulls n + 6 rows, collides n + 4 for step 1 and n
// for step 2.
//
// The arithmetic is the Walker's, operation by operation, so a pass leaves
// bit for bit the state that two single steps leave.
#pragma once

#include "lbm_device.cuh"

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

template <int S>
struct Walk2Geom {
    static constexpr int V = (S == ST_F32) ? 4 : 8;  // sites per lane, 16 bytes
    static constexpr int COLS = 30 * V;              // columns a strip stores
};

// Shared memory of one warp, in 16-byte vectors.
template <int S, int VA>
constexpr int walk2_vecs() {
    // two landing rows, rows after step 1, the row that waits for step 2's
    // collision; six rows of alpha values with a c2 field.
    return 4 * 9 * 32 + (VA ? 6 * (Walk2Geom<S>::V / 4) * 32 : 0);
}

template <int S, int LD = LD_NC, int RND = 0, int VA = 0>
struct Walker2 {
    static constexpr int V = Walk2Geom<S>::V;
    static constexpr int NW = Pack<S, V>::NW;
    static constexpr int COLS = Walk2Geom<S>::COLS;
    static_assert(NW == 4, "a lane holds one 16-byte vector per direction");
    static_assert(RND == 0 || S != ST_F32, "stochastic rounding applies to 16-bit storage");
    using T = typename StoreT<S>::T;
    uint32_t rkey1 = 0, rkey2 = 0;  // sr_step_key of the two steps
    const float *__restrict__ a15f = nullptr;

    const T *__restrict__ fin;
    T *__restrict__ fout;
    int nx, ny;
    size_t P;
    int lane, xl;
    bool act;

    __device__ __forceinline__ Walker2(const void *fin_, void *fout_, int nx_, int ny_, size_t P_,
                                       int x0)
        : fin(reinterpret_cast<const T *>(fin_)),
          fout(reinterpret_cast<T *>(fout_)),
          nx(nx_),
          ny(ny_),
          P(P_) {
        lane = threadIdx.x & 31;
        const int xu = x0 + (lane - 1) * V;  // the lane's columns, unwrapped
        act = lane >= 1 && lane <= 30 && xu < nx;
        xl = xu % nx;
        if (xl < 0) xl += nx;
    }
    __device__ __forceinline__ void set_step(uint32_t step) {
        rkey1 = sr_step_key(step);
        rkey2 = sr_step_key(step + 1u);
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
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int sr = (EYi(i) > 0) ? qm : ((EYi(i) < 0) ? qp : q0);
            const T *src = fin + ((size_t)i * P + (size_t)sr * nx + xl);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(land + i * 32)),
                         "l"(src)
                         : "memory");
        }
        if constexpr (VA) {
#pragma unroll
            for (int h = 0; h < V / 4; ++h)
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
                                            const uint4 *al) const {
        const float lft = __shfl_up_sync(FULL, d[V - 1], 1);
        const float rgt = __shfl_down_sync(FULL, d[0], 1);
        float a15v[V];
        if constexpr (VA) {
#pragma unroll
            for (int h = 0; h < V / 4; ++h) {
                const uint4 u = al[h * 32];
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
                    const uint32_t base =
                        sr_pair_base((uint32_t)r * (uint32_t)nx + (uint32_t)(xl + v), rkey);
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

    __device__ __forceinline__ void store(int r, const uint32_t (&w)[9][4]) const {
        if (!act) return;
        T *dst = fout + ((size_t)r * nx + xl);
#pragma unroll
        for (int i = 0; i < 9; ++i) store_words<S, V>(dst + (size_t)i * P, w[i]);
    }

    // Advances rows y0 .. y1-1 by two steps (two = false: by one), walking in
    // direction dir.  `buf`: the warp's walk2_vecs() vectors.
    __device__ __forceinline__ void run(int y0, int y1, int dir, bool two, const Coef &c,
                                        uint4 *buf) const {
        uint4 *land = buf + lane;  // two slots
        uint4 *wait2 = buf + 18 * 32 + lane;
        uint4 *held = buf + 27 * 32 + lane;  // [0..2]: e_y = 0 of row q - 1;
                                             // [3..5], [6..8]: the late trio of q - 1, q - 2
        uint4 *al = buf + 36 * 32 + lane;
        constexpr int AV = (V / 4) * 32;
        const float sgn = dir > 0 ? 1.f : -1.f;
        const int ext = two ? 3 : 1;
        const int K = y1 - y0 + 2 * ext;
        // The next row to copy (wrapped) and the rows before and after it.
        int q0 = (dir > 0 ? y0 - ext : y1 - 1 + ext) % ny;
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
        int row = q0;                // the pulled row
        int r1 = 0, r2 = 0, r3 = 0;  // rows pulled one, two and three iterations ago

        uint32_t wc[9][4] = {};  // the pulled row of step 1 that waits
        float d2[V], d1[V], d0[V], e2[V], e1[V], e0[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            d2[v] = d1[v] = 0.f;
            e2[v] = e1[v] = e0[v] = 0.f;
        }
        int ia = 0;  // alpha slot of the pulled row, mod 6
        issue(qm, q0, qp, land, al);
        next();
        issue(qm, q0, qp, land + 9 * 32, al + AV);  // K >= 3
        next();
        for (int k = 0; k < K; ++k) {
            uint32_t w[9][4];
            uint4 *slot = land + (k & 1) * 9 * 32;
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            take(w, slot);
            finish(w, d0);
            // The words read from the landing row have been used (the
            // shuffles), so the next copy cannot overtake them.
            if (k + 2 < K) {
                issue(qm, q0, qp, slot, al + (ia < 4 ? ia + 2 : ia - 4) * AV);
                next();
            } else {
                asm volatile("cp.async.commit_group;" ::: "memory");  // keeps the count
            }
            uint32_t u[9][4];
#pragma unroll
            for (int i = 0; i < 9; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    u[i][j] = wc[i][j];
                    wc[i][j] = w[i][j];
                }
            if (k >= 2) {
                const uint4 *a1 = al + (ia == 0 ? 5 : ia - 1) * AV;
                collide(r1, u, d1, d2, d0, sgn, c, rkey1, a1);
                if (!two) {
                    store(r1, u);
                } else {
                    // Row q after step 1 is in u.  The pulled row s = q - 1 of
                    // step 2 takes e_y = 0 from row q - 1 and, in walking
                    // order, one diagonal-and-axis trio from q and the other
                    // from q - 2.
                    uint4 *late = held + (3 + 3 * (k & 1)) * 32;
                    auto swap = [&](int i, uint4 *slot) {
                        const uint4 o = *slot;
                        *slot = make_uint4(u[i][0], u[i][1], u[i][2], u[i][3]);
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
                    if (k >= 4) {
                        finish(u, e0);
                        if (k >= 6) {
                            uint32_t z[9][4];
                            take(z, wait2);
                            keep(wait2, u);
                            const uint4 *a2 = al + (ia >= 3 ? ia - 3 : ia + 3) * AV;
                            collide(r3, z, e1, e2, e0, sgn, c, rkey2, a2);
                            store(r3, z);
                        } else {
                            keep(wait2, u);
                        }
                    }
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                d2[v] = d1[v];
                d1[v] = d0[v];
                e2[v] = e1[v];
                e1[v] = e0[v];
            }
            r3 = r2;
            r2 = r1;
            r1 = row;
            row += dir;
            if (row < 0) row += ny;
            if (row >= ny) row -= ny;
            ia = ia == 5 ? 0 : ia + 1;
        }
    }
};

}  // namespace vss

// Inner Lanczos of the nested method, per RHS (App. C steps 3-4, Eqs. popt,
// precond, innersign):
//   p      = (z_min z_max)^{-1/2}, z_max by power iteration with H_k and z_min
//            by inverse iteration with the LU of H_k (30 steps each, from the
//            normalised all-ones vector), unless p is given; with one p for
//            the batch, z_min and z_max are the extremes over its RHS (two
//            launches: the estimates of every RHS, then the rest);
//   LU of H_k in LAPACK gttrf form (partial pivoting; U with two
//            super-diagonals); the LU of p H_k has the same multipliers and
//            p times its U, so (p H_k)^{-1} x = H_k^{-1} x / p;
//   inner (two-sided) Lanczos of size l with H_k' = [p H_k + (p H_k)^{-1}]/2 and
//            e_1, applying (p H_k)^{-1} by the gttrs back substitution and
//            p H_k by a band product (App. C step 4 (a), (b)).
// In the Hermitian case (mu = 0) all of it is real arithmetic (App. C).
//
// One thread-block cluster of up to 8 CTAs per RHS.  The rows of H_k are dealt
// out in contiguous runs of R = 1..3 to the lanes of the cluster; a lane keeps
// its rows of every vector and factor in registers.  Two-sided: warps 0-1 of
// a CTA run the right recurrence (v, r), warps 2-3 the left one (w, l) side by
// side; Hermitian: four warps of the one recurrence.
//
// The substitution sweeps of gttrs are linear recurrences and run as parallel
// prefixes over affine maps:
//   first order  (L sweep with interchanges):  s <- a s + c
//   second order (U sweep, two super-diagonals): X <- M X + v, X = (x_i, x_{i+1}).
// The factor parts (a, M) of every level of the prefix depend on the LU only
// and are tabulated once; a solve composes only c and v: over the lane's
// rows, by shuffles within the warp, and from one warp aggregate per warp
// across the cluster (each warp leaves its aggregate in the shared memory of
// all CTAs; after one cluster barrier every warp combines those before it with
// tabulated products and one warp sum).  A step has four cluster barriers: after the
// first and the second sweep, and for the two inner products.
//
// What bounds it: the chain of dependent FP64 warp instructions (64 clocks
// each on GB300, whatever the active lanes) -- about 250 per step and warp at
// k = 1024, two-sided -- and the barriers.  One CTA per RHS with the vectors
// in global memory (the earlier form) ran 4 to 8 warps of 8 rows a lane on one
// SM's pipe.  Measured, this part alone: 12 two-sided RHS at k = 1024, l = 128
// 16.5 -> 4.0 ms (20 us per step, 0.9 ms for the LU, 0.5 for p); the whole inner
// part of a 6^4 solve at k = 512, l = 128 16 -> 9 ms.
#include <cooperative_groups.h>

#include "inner_arith.cuh"
#include "nk_kernels.h"

namespace cg = cooperative_groups;

namespace nk {

namespace {

constexpr int kInnerThreads = 128;
constexpr int kMaxWarps = 32;   // warps of one recurrence over the cluster

template <typename T> struct IsC { static constexpr bool value = false; };
template <> struct IsC<double2> { static constexpr bool value = true; };

// Sums over the lanes of a warp, the result in every lane; real and imaginary
// parts (and the two components of a second-order state) share the levels of
// the butterfly, one FP64 addition each.
__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ double2 warp_total(double2 v) {
    const bool up = (threadIdx.x & 16) != 0;
    double t = (up ? v.y : v.x) + __shfl_xor_sync(kFull, up ? v.x : v.y, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    return mk(__shfl_sync(kFull, t, 0), __shfl_sync(kFull, t, 16));
}
__device__ __forceinline__ void warp_total2(double& a, double& b) {
    const double2 t = warp_total(mk(a, b));
    a = t.x;
    b = t.y;
}
__device__ __forceinline__ void warp_total2(double2& a, double2& b) {
    const bool up = (threadIdx.x & 16) != 0, im = (threadIdx.x & 8) != 0;
    double2 t = up ? b : a;
    const double2 o = up ? a : b;
    t.x += __shfl_xor_sync(kFull, o.x, 16);
    t.y += __shfl_xor_sync(kFull, o.y, 16);
    double s = (im ? t.y : t.x) + __shfl_xor_sync(kFull, im ? t.x : t.y, 8);
#pragma unroll
    for (int l = 4; l > 0; l >>= 1) s += __shfl_xor_sync(kFull, s, l);
    a = mk(__shfl_sync(kFull, s, 0), __shfl_sync(kFull, s, 8));
    b = mk(__shfl_sync(kFull, s, 16), __shfl_sync(kFull, s, 24));
}

// Tridiagonal LU with partial pivoting, LAPACK gttrf semantics (rows i and
// i + 1 are interchanged when |d_i| < |dl_i|, |.| = |re| + |im| for complex), by
// one warp: all lanes run the recurrence, lane t keeps row c0 + t of each chunk
// of 32 rows; the diagonals of the chunk and the inverses of its subdiagonal
// (the pivots of interchanged rows) are prepared by lane in shared memory (buf,
// 4 x 32).  Writes the multipliers dl, the rows du, du2 of U, dinv = 1/d and
// the interchanges piv (1: rows i and i + 1).  Returns 0, or i + 1 if U(i,i) = 0.
template <typename T>
__device__ int gttrf_warp(int n, const double2* al, const double2* be, const double2* ga, T* dl, T* dinv, T* du,
                          T* du2, int* piv, T* buf) {
    const int lane = threadIdx.x & 31;
    T *bB = buf, *bA = buf + 32, *bG = buf + 64, *bI = buf + 96;
    T d = t_from(al[0], T()), u = t_from(ga[0], T());
    int info = 0;
    for (int c0 = 0; c0 < n; c0 += 32) {
        const int row = c0 + lane;
        const T b = row < n - 1 ? t_from(be[row], T()) : t_zero(T());
        __syncwarp();
        bB[lane] = b;
        bA[lane] = row < n - 1 ? t_from(al[row + 1], T()) : t_zero(T());
        bG[lane] = row < n - 2 ? t_from(ga[row + 1], T()) : t_zero(T());
        bI[lane] = t_iszero(b) ? t_zero(T()) : pivot_div(b);
        __syncwarp();
        T o_dl = t_zero(T()), o_di = t_zero(T()), o_du = t_zero(T()), o_du2 = t_zero(T());
        int o_pv = 0;
        const int m = min(32, n - c0);
        for (int t = 0; t < m; ++t) {
            const T Bt = bB[t], At = bA[t], Gt = bG[t], It = bI[t];
            const bool zero = t_iszero(d), lastrow = c0 + t == n - 1;
            const bool keep = lastrow || t_abs1(d) >= t_abs1(Bt);
            T fact, pd, pu, pu2, inv;
            if (keep) {
                inv = zero ? t_zero(T()) : pivot_div(d);
                fact = zero ? Bt : t_mul(Bt, inv);   // d = 0 only with a zero subdiagonal
                pd = d;
                pu = u;
                pu2 = t_zero(T());
                d = zero ? At : t_fma(t_neg(fact), u, At);
                u = Gt;
            } else {
                inv = It;
                fact = t_mul(d, It);
                pd = Bt;
                pu = At;
                pu2 = Gt;
                d = t_fma(t_neg(fact), At, u);
                u = t_mul(t_neg(fact), Gt);
            }
            if (t_iszero(pd) && !info) info = c0 + t + 1;
            if (lane == t) {
                o_dl = fact;
                o_di = inv;
                o_du = pu;
                o_du2 = pu2;
                o_pv = keep ? 0 : 1;
            }
        }
        if (row < n) {
            dl[row] = o_dl;
            dinv[row] = o_di;
            du[row] = o_du;
            du2[row] = o_du2;
            piv[row] = o_pv;
        }
    }
    return info;
}

// Shared memory of a CTA.  Tables [row][thread]; buffers by warp of the
// recurrence over the cluster (group g of the two recurrences).
template <typename T>
struct InnerSmem {
    T tab1[6][kInnerThreads];     // a before each shuffle level; 5: a of the intra-warp exclusive prefix
    T tab2[24][kInnerThreads];    // M before each level (4 entries each); 20-23: of the exclusive prefix
    T crs1[kInnerThreads];        // product of the a of the warps between warp q = lane and this one
    T crs2[4][kInnerThreads];     // the same of M
    T agg[4][2][kMaxWarps][2];    // warp aggregates: sweep 1, sweep 2, inner product 1, inner product 2
    T halo[2][kMaxWarps][2];      // first and last row of each warp's v (w)
    T sw[3 * 128];                // w of the CTA's rows
    T sr[3 * 128];                // r
    T lu[4 * 32];                 // gttrf_warp
    double flag;
};

// phase 0: p of this RHS, then steps 3-4.  With a p shared by the batch
// (Inner::p_shared) two launches: phase 1 estimates z_min, z_max of every RHS
// and stops (its LU stays in the work area); phase 2 takes p from the extremes
// over the batch and runs steps 3-4 with that LU.
template <typename T, int R>
__global__ void __launch_bounds__(kInnerThreads) k_inner(Inner in, int phase, int C) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    InnerSmem<T>& S = *reinterpret_cast<InnerSmem<T>*>(smem_raw);
    constexpr bool TS = IsC<T>::value;
    constexpr int WG = TS ? 2 : 4;            // warps of one recurrence per CTA
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int rhs = blockIdx.x / C;
    const int n = in.k, L = in.ell;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = warp / WG, gw = warp % WG;  // recurrence (0 right, 1 left), warp in it
    const int NW = C * WG, W = rank * WG + gw;
    const int lo = (W * 32 + lane) * R;       // this lane's rows [lo, lo + R)
    const int loc = (gw * 32 + lane) * R;     // the same within the CTA
    const int status0 = in.status[rhs];
    cl.sync();   // every CTA has read the status (and is resident) before anything is written
    if (status0 != kStatusOK) {
        // no estimate from this RHS (a frozen RHS of adaptive k keeps the one
        // from the H_k it converged with)
        if (phase == 1 && rank == 0 && tid == 0 && status0 != kStatusConverged) {
            in.zmin[rhs] = 0.0;
            in.zmax[rhs] = 0.0;
        }
        return;
    }
    const int ks = in.kstride > 0 ? in.kstride : n;   // row stride of the outer H_k arrays and of c
    const double2* gal = in.alpha + (size_t)rhs * ks;
    const double2* gbe = in.beta + (size_t)rhs * ks;
    const double2* gga = in.gamma + (size_t)rhs * ks;
    T* wk = reinterpret_cast<T*>(in.work + (size_t)rhs * inner_work_elems(n));
    T *w_dl = wk, *w_di = wk + n, *w_du = wk + 2 * n, *w_du2 = wk + 3 * n;
    double* w_info = reinterpret_cast<double*>(wk + 4 * n);
    int* w_pv = in.ipiv + (size_t)rhs * n;

    // value `val` (the same in every lane) into `slot` of every CTA
    auto pub = [&](T* slot, T val) {
        if (lane < C) *cl.map_shared_rank(slot, lane) = val;
    };
    auto live = [&](int t) { return lo + t < n; };

    // ---- LU of H_k (rank 0; phase 2 finds it in the work area) --------------------
    if (phase != 2 && rank == 0 && warp == 0) {
        const int info = gttrf_warp<T>(n, gal, gbe, gga, w_dl, w_di, w_du, w_du2, w_pv, S.lu);
        if (lane == 0) *w_info = (double)info;
        __threadfence();
    }
    cl.sync();
    const bool singular = __ldcg(w_info) != 0.0;

    // band entries and factors of this lane's rows.  Right: A1 = dl_{i-1},
    // e2 = -du_i/d_i, f2 = -du2_i/d_i; left: A1 = dl_i^*, e2 = -(du_{i-1}/d_i)^*,
    // f2 = -(du2_{i-2}/d_i)^*, and everything else conjugated.  Bits of `swp`: row i
    // interchanged with i + 1; of `swm`: row i - 1 with i.
    T al[R], sub[R], sup[R], A1[R], e2[R], f2[R], di[R];
    T A1m = t_zero(T());   // left: dl_{lo-1}^*
    unsigned swp = 0, swm = 0;
    auto ld = [&](const T* p, int i) { return i >= 0 && i < n ? p[i] : t_zero(T()); };
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int i = lo + t;
        al[t] = sub[t] = sup[t] = A1[t] = e2[t] = f2[t] = di[t] = t_zero(T());
        if (i >= n) continue;
        T a = t_from(gal[i], T()), b = i > 0 ? t_from(gbe[i - 1], T()) : t_zero(T());
        T c = i < n - 1 ? t_from(gga[i], T()) : t_zero(T());
        if (g == 1) {
            const T s = i > 0 ? t_from(gga[i - 1], T()) : t_zero(T());
            c = i < n - 1 ? t_conj(t_from(gbe[i], T())) : t_zero(T());
            b = t_conj(s);
            a = t_conj(a);
        }
        al[t] = a;
        sub[t] = b;
        sup[t] = c;
        const T dv = __ldcg(w_di + i);
        if (i < n - 1 && __ldcg(w_pv + i)) swp |= 1u << t;
        if (i > 0 && __ldcg(w_pv + i - 1)) swm |= 1u << t;
        if (g == 0) {
            A1[t] = i > 0 ? __ldcg(w_dl + i - 1) : t_zero(T());
            e2[t] = i < n - 1 ? t_neg(t_mul(__ldcg(w_du + i), dv)) : t_zero(T());
            f2[t] = i < n - 2 ? t_neg(t_mul(__ldcg(w_du2 + i), dv)) : t_zero(T());
            di[t] = dv;
        } else {
            A1[t] = i < n - 1 ? t_conj(__ldcg(w_dl + i)) : t_zero(T());
            if (t == 0 && i > 0) A1m = t_conj(__ldcg(w_dl + i - 1));
            e2[t] = i > 0 ? t_neg(t_conj(t_mul(__ldcg(w_du + i - 1), dv))) : t_zero(T());
            f2[t] = i > 1 ? t_neg(t_conj(t_mul(__ldcg(w_du2 + i - 2), dv))) : t_zero(T());
            di[t] = t_conj(dv);
        }
    }

    // ---- prefix machinery -----------------------------------------------------------
    // direction of this recurrence's sweeps: the right one runs L ascending and
    // U descending, the left one U^dagger ascending and L^dagger descending
    const bool asc1 = g == 0, asc2 = g == 1;
    auto dirsh = [&](T v, int o, bool asc) { return asc ? shup(v, o) : shdn(v, o); };
    auto partner = [&](int o, bool asc) { return asc ? lane >= o : lane + o < 32; };
    auto firstl = [&](bool asc) { return asc ? lane == 0 : lane == 31; };
    auto pos = [&](bool asc) { return asc ? W : NW - 1 - W; };
    auto at = [&](int q, bool asc) { return asc ? q : NW - 1 - q; };   // warp at position q

    // first-order map of row t applied to s, with right-hand side b:
    // not interchanged b - dl s, interchanged s - dl b (right) or s (left)
    auto map1 = [&](int t, T s, T b) -> T {
        const int i = lo + t;
        if (i >= n) return s;
        if (g == 0) {
            if (i == 0) return b;
            return (swm >> t & 1) ? t_fma(t_neg(A1[t]), b, s) : t_fma(t_neg(A1[t]), s, b);
        }
        if (i == n - 1) return b;
        return (swp >> t & 1) ? s : t_fma(t_neg(A1[t]), s, b);
    };
    auto fac1 = [&](int t, T a) -> T {   // its factor part applied to a
        const int i = lo + t;
        if (i >= n) return a;
        if (i == (g == 0 ? 0 : n - 1)) return t_zero(T());
        const unsigned sw = g == 0 ? swm : swp;
        return (sw >> t & 1) ? a : t_neg(t_mul(A1[t], a));
    };

    // tables of this LU
    {
        T a = t_one(T());
        T m00 = t_one(T()), m01 = t_zero(T()), m10 = t_zero(T()), m11 = t_one(T());
        auto step2 = [&](int t) {
            if (!live(t)) return;
            const T x0 = t_fma(e2[t], m00, t_mul(f2[t], m10)), x1 = t_fma(e2[t], m01, t_mul(f2[t], m11));
            m10 = m00;
            m11 = m01;
            m00 = x0;
            m01 = x1;
        };
        if (g == 0) {
#pragma unroll
            for (int t = 0; t < R; ++t) a = fac1(t, a);
#pragma unroll
            for (int t = R - 1; t >= 0; --t) step2(t);
        } else {
#pragma unroll
            for (int t = R - 1; t >= 0; --t) a = fac1(t, a);
#pragma unroll
            for (int t = 0; t < R; ++t) step2(t);
        }
#pragma unroll 1
        for (int lv = 0, o = 1; o < 32; ++lv, o <<= 1) {
            S.tab1[lv][tid] = a;
            const T pa = dirsh(a, o, asc1);
            if (partner(o, asc1)) a = t_mul(a, pa);
            S.tab2[4 * lv][tid] = m00;
            S.tab2[4 * lv + 1][tid] = m01;
            S.tab2[4 * lv + 2][tid] = m10;
            S.tab2[4 * lv + 3][tid] = m11;
            const T p00 = dirsh(m00, o, asc2), p01 = dirsh(m01, o, asc2), p10 = dirsh(m10, o, asc2),
                    p11 = dirsh(m11, o, asc2);
            if (partner(o, asc2)) {
                const T n00 = t_fma(m00, p00, t_mul(m01, p10)), n01 = t_fma(m00, p01, t_mul(m01, p11));
                const T n10 = t_fma(m10, p00, t_mul(m11, p10)), n11 = t_fma(m10, p01, t_mul(m11, p11));
                m00 = n00;
                m01 = n01;
                m10 = n10;
                m11 = n11;
            }
        }
        const T ea = dirsh(a, 1, asc1);
        S.tab1[5][tid] = firstl(asc1) ? t_one(T()) : ea;
        const T e00 = dirsh(m00, 1, asc2), e01 = dirsh(m01, 1, asc2), e10 = dirsh(m10, 1, asc2), e11 = dirsh(m11, 1, asc2);
        const bool f2l = firstl(asc2);
        S.tab2[20][tid] = f2l ? t_one(T()) : e00;
        S.tab2[21][tid] = f2l ? t_zero(T()) : e01;
        S.tab2[22][tid] = f2l ? t_zero(T()) : e10;
        S.tab2[23][tid] = f2l ? t_one(T()) : e11;
        const int l1 = asc1 ? 31 : 0, l2 = asc2 ? 31 : 0;
        pub(&S.agg[0][g][W][0], shfl_from(a, l1));
        pub(&S.agg[1][g][W][0], shfl_from(m00, l2));
        pub(&S.agg[1][g][W][1], shfl_from(m01, l2));
        pub(&S.agg[2][g][W][0], shfl_from(m10, l2));
        pub(&S.agg[2][g][W][1], shfl_from(m11, l2));
        cl.sync();
        // products over the warps strictly between position q = lane and this warp's
        a = t_one(T());
        m00 = m11 = t_one(T());
        m01 = m10 = t_zero(T());
        const int p1 = pos(asc1), p2 = pos(asc2);
#pragma unroll 1
        for (int s = 1; s < NW; ++s) {
            const int w1 = at(s, asc1), w2 = at(s, asc2);
            if (s > lane && s < p1) a = t_mul(S.agg[0][g][w1][0], a);
            if (s > lane && s < p2) {
                const T g00 = S.agg[1][g][w2][0], g01 = S.agg[1][g][w2][1], g10 = S.agg[2][g][w2][0],
                        g11 = S.agg[2][g][w2][1];
                const T n00 = t_fma(g00, m00, t_mul(g01, m10)), n01 = t_fma(g00, m01, t_mul(g01, m11));
                const T n10 = t_fma(g10, m00, t_mul(g11, m10)), n11 = t_fma(g10, m01, t_mul(g11, m11));
                m00 = n00;
                m01 = n01;
                m10 = n10;
                m11 = n11;
            }
        }
        S.crs1[tid] = a;
        S.crs2[0][tid] = m00;
        S.crs2[1][tid] = m01;
        S.crs2[2][tid] = m10;
        S.crs2[3][tid] = m11;
        cl.sync();   // the aggregates have been read everywhere
    }

    // Sweep in two halves around a cluster barrier: the composition of the
    // lane's rows and the warp, whose aggregate goes to every CTA (buffer b) ...
    auto first_begin = [&](const T (&x)[R], int b) -> T {
        T c = t_zero(T());
        if (g == 0) {
#pragma unroll
            for (int t = 0; t < R; ++t) c = map1(t, c, x[t]);
        } else {
#pragma unroll
            for (int t = R - 1; t >= 0; --t) c = map1(t, c, x[t]);
        }
#pragma unroll
        for (int lv = 0, o = 1; o < 32; ++lv, o <<= 1) {
            const T pc = dirsh(c, o, asc1);
            if (partner(o, asc1)) c = t_fma(S.tab1[lv][tid], pc, c);
        }
        pub(&S.agg[b][g][W][0], shfl_from(c, asc1 ? 31 : 0));
        const T ex = dirsh(c, 1, asc1);
        return firstl(asc1) ? t_zero(T()) : ex;
    };
    // ... and the state that enters the lane's rows
    auto first_end = [&](T cex, int b) -> T {
        const int p = pos(asc1);
        T v = t_zero(T());
        if (lane < p) v = t_mul(S.crs1[tid], S.agg[b][g][at(lane, asc1)][0]);
        return t_fma(S.tab1[5][tid], warp_total(v), cex);
    };
    auto second_begin = [&](const T (&yd)[R], int b, T& v0, T& v1) {
        v0 = v1 = t_zero(T());
        auto row = [&](int t) {
            if (!live(t)) return;
            const T x = t_fma(e2[t], v0, t_fma(f2[t], v1, yd[t]));
            v1 = v0;
            v0 = x;
        };
        if (g == 0) {
#pragma unroll
            for (int t = R - 1; t >= 0; --t) row(t);
        } else {
#pragma unroll
            for (int t = 0; t < R; ++t) row(t);
        }
#pragma unroll
        for (int lv = 0, o = 1; o < 32; ++lv, o <<= 1) {
            const T p0 = dirsh(v0, o, asc2), p1 = dirsh(v1, o, asc2);
            if (partner(o, asc2)) {
                v0 = t_fma(S.tab2[4 * lv][tid], p0, t_fma(S.tab2[4 * lv + 1][tid], p1, v0));
                v1 = t_fma(S.tab2[4 * lv + 2][tid], p0, t_fma(S.tab2[4 * lv + 3][tid], p1, v1));
            }
        }
        const int ll = asc2 ? 31 : 0;
        pub(&S.agg[b][g][W][0], shfl_from(v0, ll));
        pub(&S.agg[b][g][W][1], shfl_from(v1, ll));
        const T x0 = dirsh(v0, 1, asc2), x1 = dirsh(v1, 1, asc2);
        const bool f = firstl(asc2);
        v0 = f ? t_zero(T()) : x0;
        v1 = f ? t_zero(T()) : x1;
    };
    auto second_end = [&](int b, T& v0, T& v1) {
        const int p = pos(asc2);
        T u0 = t_zero(T()), u1 = t_zero(T());
        if (lane < p) {
            const int w = at(lane, asc2);
            const T a0 = S.agg[b][g][w][0], a1 = S.agg[b][g][w][1];
            u0 = t_fma(S.crs2[0][tid], a0, t_mul(S.crs2[1][tid], a1));
            u1 = t_fma(S.crs2[2][tid], a0, t_mul(S.crs2[3][tid], a1));
        }
        warp_total2(u0, u1);
        v0 = t_fma(S.tab2[20][tid], u0, t_fma(S.tab2[21][tid], u1, v0));
        v1 = t_fma(S.tab2[22][tid], u0, t_fma(S.tab2[23][tid], u1, v1));
    };
    // the first and last row of this warp's x to every CTA
    auto pub_halo = [&](const T (&x)[R]) {
        pub(&S.halo[g][W][0], shfl_from(x[0], 0));
        pub(&S.halo[g][W][1], shfl_from(x[R - 1], 31));
    };
    auto next_of = [&](const T (&x)[R]) -> T {   // x_{lo + R}, after the barrier of pub_halo
        T v = shdn(x[0], 1);
        if (lane == 31) v = W < NW - 1 ? S.halo[g][W + 1][0] : t_zero(T());
        return v;
    };
    auto prev_of = [&](const T (&x)[R]) -> T {   // x_{lo - 1}
        T v = shup(x[R - 1], 1);
        if (lane == 0) v = W > 0 ? S.halo[g][W - 1][1] : t_zero(T());
        return v;
    };
    // y = H x (left: H^dagger x)
    auto band = [&](const T (&x)[R], T (&y)[R]) {
        const T xm = prev_of(x), xp = next_of(x);
#pragma unroll
        for (int t = 0; t < R; ++t)
            y[t] = t_fma(sup[t], t + 1 < R ? x[t + 1] : xp, t_fma(sub[t], t > 0 ? x[t - 1] : xm, t_mul(al[t], x[t])));
    };
    // y = H^{-1} x (left: (H^dagger)^{-1} x): begins with a barrier that also
    // completes pub_halo(x), and holds a second one
    auto solve = [&](const T (&x)[R], T (&y)[R]) {
        T yd[R], c1, v0, v1;
        if (g == 0) {
            c1 = first_begin(x, 0);
        } else {
#pragma unroll
            for (int t = 0; t < R; ++t) yd[t] = t_mul(x[t], di[t]);
            second_begin(yd, 0, v0, v1);
        }
        cl.sync();
        if (g == 0) {
            T s = first_end(c1, 0);
            const T xp = next_of(x);
#pragma unroll
            for (int t = 0; t < R; ++t) {
                s = map1(t, s, x[t]);
                const T nx = t + 1 < R ? x[t + 1] : xp;
                yd[t] = t_mul((swp >> t & 1) ? nx : s, di[t]);
            }
            second_begin(yd, 1, v0, v1);
        } else {
            second_end(0, v0, v1);
            const T x_lo = v0;   // the U^dagger result of row lo - 1
#pragma unroll
            for (int t = 0; t < R; ++t) {
                if (!live(t)) { y[t] = t_zero(T()); continue; }
                const T z = t_fma(e2[t], v0, t_fma(f2[t], v1, yd[t]));
                v1 = v0;
                v0 = z;
                y[t] = z;
            }
            c1 = first_begin(y, 1);
            v0 = x_lo;
        }
        cl.sync();
        if (g == 0) {
            second_end(1, v0, v1);
#pragma unroll
            for (int t = R - 1; t >= 0; --t) {
                if (!live(t)) { y[t] = t_zero(T()); continue; }
                const T z = t_fma(e2[t], v0, t_fma(f2[t], v1, yd[t]));
                v1 = v0;
                v0 = z;
                y[t] = z;
            }
        } else {
            T s = first_end(c1, 1);
#pragma unroll
            for (int t = R - 1; t >= 0; --t) {
                if (!live(t)) continue;
                s = map1(t, s, y[t]);
                // row i - 1 interchanged: in_{i-1} - dl_{i-1}^* s_i, else s_i
                const T in_m = t > 0 ? y[t - 1] : v0, dl_m = t > 0 ? A1[t - 1] : A1m;
                y[t] = (swm >> t & 1) ? t_fma(t_neg(dl_m), s, in_m) : s;
            }
        }
    };
    // sum over the rows of a group's lanes, to every thread (buffer 2 or 3):
    // the group publishes, one barrier, then everyone adds the NW warp sums
    auto sum_begin = [&](T part, int b) {
        const T t = warp_total(part);
        pub(&S.agg[b][g][W][0], t);
    };
    auto sum_end = [&](int b, int from) -> T {
        return warp_total(lane < NW ? S.agg[b][from][lane][0] : t_zero(T()));
    };
    // |x| of the right group's x in every thread (one barrier)
    auto norm = [&](const T (&x)[R]) -> double {
        if (g == 0) {
            double s = 0.0;
#pragma unroll
            for (int t = 0; t < R; ++t) s += t_norm2(x[t]);
            s = warp_total(s);
            pub(&S.agg[2][0][W][0], t_from(mk(s, 0.0), T()));
        }
        cl.sync();
        return sqrt(warp_total(lane < NW ? t_to2(S.agg[2][0][lane][0]).x : 0.0));
    };

    // ---- p (Eq. popt) --------------------------------------------------------
    double p = in.p_fixed;
    if (!(p > 0.0) && phase == 2) {
        // Eq. popt with z_min = min |z| and z_max = max |z| of A, estimated as
        // the extremes over the batch's H_k (all RHS share A); every CTA forms
        // the same value in the same order
        double zmn = 0.0, zmx = 0.0;
        for (int r = 0; r < in.n_rhs; ++r) {
            const double a = in.zmin[r], b = in.zmax[r];
            if (a > 0.0 && b > 0.0 && isfinite(a) && isfinite(b)) {
                zmn = zmn > 0.0 ? fmin(zmn, a) : a;
                zmx = fmax(zmx, b);
            }
        }
        p = zmn > 0.0 ? 1.0 / sqrt(zmn * zmx) : 1.0;
    } else if (!(p > 0.0)) {
        const double x0 = 1.0 / sqrt((double)n);
        T x[R], y[R];
        auto start = [&] {
#pragma unroll
            for (int t = 0; t < R; ++t) x[t] = live(t) ? t_from(mk(x0, 0.0), T()) : t_zero(T());
        };
        auto rescale = [&](double s) {
#pragma unroll
            for (int t = 0; t < R; ++t) x[t] = t_scale(y[t], s);
        };
        start();
        double zmax = 0.0;
        for (int it = 0; it < 30; ++it) {
            pub_halo(x);
            cl.sync();
            band(x, y);
            zmax = norm(y);
            rescale(1.0 / zmax);
        }
        // inverse iteration with the LU of H itself (both groups run it; the
        // right one's result counts)
        start();
        double tn = 1.0;
        for (int it = 0; it < 30; ++it) {
            pub_halo(x);
            solve(x, y);
            tn = norm(y);
            rescale(1.0 / tn);
        }
        double zmin = 1.0 / tn;
        // Accept the smallest Ritz value only if its Ritz pair has converged
        // (residual |H(k-1,k-2)| |x_{k-1}| <= 0.1 z); otherwise it is a spurious
        // value in the spectral gap: iterate again with that direction projected out.
        if (g == 0) {
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (lo + t == n - 1)
                    for (int q = 0; q < C; ++q)
                        *cl.map_shared_rank(&S.flag, q) = sqrt(cnorm2(gbe[n - 2])) * sqrt(t_norm2(x[t]));
        }
        cl.sync();
        const double resid = S.flag;
        if (resid > 0.1 * zmin) {
            T x1[R];
#pragma unroll
            for (int t = 0; t < R; ++t) x1[t] = x[t];
            // a <- a - (x1^dag a) x1 (x1 of unit norm), the right group's a
            auto project = [&](T (&a)[R]) {
                T d = t_zero(T());
#pragma unroll
                for (int t = 0; t < R; ++t) d = t_dot_add(d, x1[t], a[t]);
                if (g == 0) sum_begin(d, 3);
                cl.sync();
                d = t_neg(sum_end(3, 0));
#pragma unroll
                for (int t = 0; t < R; ++t) a[t] = t_fma(d, x1[t], a[t]);
            };
            start();
            project(x);
            const double xn = 1.0 / norm(x);
#pragma unroll
            for (int t = 0; t < R; ++t) x[t] = t_scale(x[t], xn);
            for (int it = 0; it < 30; ++it) {
                pub_halo(x);
                solve(x, y);
                project(y);
                tn = norm(y);
                rescale(1.0 / tn);
            }
            zmin = 1.0 / tn;
        }
        p = 1.0 / sqrt(zmin * zmax);
        if (rank == 0 && tid == 0) { in.zmin[rhs] = zmin; in.zmax[rhs] = zmax; }
        if (phase == 1) return;
    } else if (rank == 0 && tid == 0) {
        in.zmin[rhs] = 0.0; in.zmax[rhs] = 0.0;
    }
    if (rank == 0 && tid == 0) in.p[rhs] = p;
    if (singular) {
        if (rank == 0 && tid == 0) in.status[rhs] = kStatusLU;
        return;
    }

    // ---- step 4: inner (two-sided) Lanczos with H' and e_1 ----------------------
    // v (left: w), the vector before it and r (left: l), this lane's rows
    T v[R], vp[R], r[R], x[R];
#pragma unroll
    for (int t = 0; t < R; ++t) {
        v[t] = lo + t == 0 ? t_one(T()) : t_zero(T());
        vp[t] = t_zero(T());
    }
    const double hp = 0.5 * p, hi = 0.5 / p;
    double2* Vl = in.Vl + (size_t)rhs * L * n;
    double2* alo = in.al + (size_t)rhs * L;
    double2* blo = in.bl + (size_t)rhs * L;
    double2* glo = in.gl + (size_t)rhs * L;
    const bool first = rank == 0 && tid == 0;
    T back = t_zero(T());   // gamma_{j-1} (left: beta_{j-1}^*)
    for (int j = 0; j < L; ++j) {
        if (g == 0) {
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (live(t)) Vl[(size_t)j * n + lo + t] = t_to2(v[t]);
        } else {
#pragma unroll
            for (int t = 0; t < R; ++t) S.sw[loc + t] = v[t];
        }
        // r <- H' v - gamma v_{j-1}, H' v = [p H v + (p H)^{-1} v]/2 (left: H'^dagger)
        pub_halo(v);
        solve(v, x);
        band(v, r);
#pragma unroll
        for (int t = 0; t < R; ++t) {
            r[t] = t_add(t_scale(r[t], hp), t_scale(x[t], hi));
            if (j > 0) r[t] = t_fma(t_neg(back), vp[t], r[t]);
        }
        // H(j,j) <- v^dag r (two-sided: w^dag r)
        if (g == 0) {
            T d = t_zero(T());
#pragma unroll
            for (int t = 0; t < R; ++t) d = t_dot_add(d, TS ? S.sw[loc + t] : v[t], r[t]);
            sum_begin(d, 2);
        }
        cl.sync();
        const T a = sum_end(2, 0);
        if (first) alo[j] = t_to2(a);
        const T na = t_neg(g == 0 ? a : t_conj(a));
#pragma unroll
        for (int t = 0; t < R; ++t) r[t] = t_fma(na, v[t], r[t]);
        if (j == L - 1) break;
        if (TS) {
            if (g == 0) {
#pragma unroll
                for (int t = 0; t < R; ++t) S.sr[loc + t] = r[t];
            }
            __syncthreads();
            if (g == 1) {      // delta <- r^dag l
                T d = t_zero(T());
#pragma unroll
                for (int t = 0; t < R; ++t) d = t_dot_add(d, S.sr[loc + t], r[t]);
                sum_begin(d, 3);
            }
        } else {               // beta^2 <- r^T r
            T d = t_zero(T());
#pragma unroll
            for (int t = 0; t < R; ++t) d = t_dot_add(d, r[t], r[t]);
            sum_begin(d, 3);
        }
        cl.sync();
        const double2 d2 = t_to2(sum_end(3, TS ? 1 : 0));
        double2 b, gm, ib, ig;
        if (!TS) {
            double inv = 0.0;
            const double bb = d2.x > 0.0 && isfinite(d2.x) ? sqrt_inv(d2.x, inv) : d2.x;
            if (!(bb > 0.0)) { if (first) in.status[rhs] = kStatusInnerBreakdown; return; }
            b = gm = mk(bb, 0.0);
            ib = ig = mk(inv, 0.0);
        } else {
            if ((d2.x == 0.0 && d2.y == 0.0) || !isfinite(d2.x) || !isfinite(d2.y)) {
                if (first) in.status[rhs] = kStatusInnerBreakdown;
                return;
            }
            csqrt_scalars(d2, b, gm, ib, ig);
        }
        if (first) { blo[j] = b; glo[j] = gm; }
        // v <- r / beta, w <- l / gamma^*
        const T sc = t_from(g == 0 ? ib : cconj(ig), T());
        back = t_from(g == 0 ? gm : cconj(b), T());
#pragma unroll
        for (int t = 0; t < R; ++t) {
            vp[t] = v[t];
            v[t] = t_mul(r[t], sc);
        }
    }
}

template <typename T, int R>
cudaError_t launch_r(const Inner& in, int phase, int C, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(in.n_rhs * C));
    cfg.blockDim = dim3(kInnerThreads);
    cfg.dynamicSmemBytes = sizeof(InnerSmem<T>);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_inner<T, R>, in, phase, C);
}

// One row per lane while the cluster has lanes enough (64 a CTA two-sided, 128
// Hermitian), with the smallest cluster that does it; above 8 CTAs 2 or 3 rows.
template <typename T>
cudaError_t launch_t(const Inner& in, int phase, cudaStream_t st) {
    const int lanes = IsC<T>::value ? 64 : 128;
    int C = 1;
    while (C < 8 && C * lanes < in.k) C *= 2;
    const int R = (in.k + C * lanes - 1) / (C * lanes);
    if (R == 1) return launch_r<T, 1>(in, phase, C, st);
    if (R == 2) return launch_r<T, 2>(in, phase, C, st);
    return launch_r<T, 3>(in, phase, C, st);
}

}  // namespace

static_assert(kMaxInnerK <= 3 * 8 * 64, "at most three rows per lane of an 8-CTA cluster");
static_assert(kInnerWorkVecs >= 5, "multipliers, 1/d, du, du2 and the singularity flag");

int launch_inner_lanczos(const Inner& in, cudaStream_t st) {
    const bool shared = in.p_shared && !(in.p_fixed > 0.0);
    for (int phase = shared ? 1 : 0; phase <= (shared ? 2 : 0); ++phase) {
        const cudaError_t e = in.two_sided ? launch_t<double2>(in, phase, st) : launch_t<double>(in, phase, st);
        if (e != cudaSuccess) return (int)e;
    }
    return 0;
}

void inner_lanczos_init_attributes() {
#define NK_ATTR(T_, R_) \
    cudaFuncSetAttribute(k_inner<T_, R_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(InnerSmem<T_>))
    NK_ATTR(double, 1); NK_ATTR(double, 2); NK_ATTR(double, 3);
    NK_ATTR(double2, 1); NK_ATTR(double2, 2); NK_ATTR(double2, 3);
#undef NK_ATTR
}

}  // namespace nk

// FP64 Wilson stencil A = gamma5 D_w(mu), A^dagger = gamma5 D_w(-mu) (Sec. 2):
// alone, and fused with the first half of an outer Lanczos step.
//
// What bounds it.  A site and vector take 888 FP64 instructions per lane
// (projection 96, link products 576, accumulation and output 216), and GB300
// issues two FP64 lanes per clock and SM: one thread per site and vector
// keeps a warp on the FP64 pipe for at least 888 x 16 clocks, and on the
// small lattices most of the chip has no warp at all (4^4, one vector: 55 us
// in two CTAs; 10^4, both sides of one source: 82 us against a floor of 29).
// So a site is spread over 16 threads, one per hop h = 0..7 (nu = h / 2, odd
// h forward) and half-spinor column c: each projects its column of the
// neighbour spinor (6 additions), multiplies it by the link (36 fused
// multiply-adds) and leaves the three colours in shared memory; after one
// barrier 12 threads per site sum the eight hops of one spin-colour
// component each.  No FP64 operation is done twice, the sums run over the
// hops in the order 0..7, and a CTA of S sites (S = 4, 8 or 16) is short
// enough to fill the chip from 4^4 on.  Measured, outer step (this kernel and
// step 2) of one source: 4^4, mu = 0 51.5 -> 16.8 us (13.5 with the present step 2); 6^4,
// mu = 0.1 58 -> 28 (21); 10^4, mu = 0.2 95 -> 65 (58).  The stencil alone
// on 12 vectors at 16^3 x 32, 2.44 -> 2.34 ms (its FP64 floor is 2.25), and
// straight from and to the ABI layout, without the two conversion passes
// (0.2 ms).  Profile at 10^4: FP64 pipe 82% busy while an SM has work.
//
// The gamma matrices act on the half spinors as multiplications by i^q (swaps
// and sign flips on the integer pipe), so the lanes of a warp may work on
// different hops without diverging.  SPLIT = 3 (a launch shape) gives each
// colour row of the product its own thread: a third of the chain per thread
// for 22% more FP64 work (the projection is repeated); it was never faster at
// the default S = 8 (6^4 28 against 32 us) and level with it at S = 4, 4^4.
#include <algorithm>

#include "nk_common.cuh"
#include "nk_kernels.h"
#include "nk_step.cuh"

namespace nk {

namespace {

constexpr int kS64Sites = 56;   // sites resident per SM: 56 / S CTAs (28 warps at 72 registers)

__device__ __forceinline__ double flip(double x, unsigned mask) {   // mask: 0 or the sign bit
    return __hiloint2double(__double2hiint(x) ^ (int)mask, __double2loint(x));
}
// z * i^q
__device__ __forceinline__ double2 rot(double2 z, int q) {
    const unsigned sx = ((q + 1) & 2) ? 0x80000000u : 0u;   // q = 1, 2
    const unsigned sy = (q & 2) ? 0x80000000u : 0u;         // q = 2, 3
    const double x = (q & 1) ? z.y : z.x, y = (q & 1) ? z.x : z.y;
    return make_double2(flip(x, sx), flip(y, sy));
}

// Index of component c of a site: [12][V] (device layout) or [V][12] (ABI layout).
template <bool ABI>
__device__ __forceinline__ size_t comp_at(int c, int site, int V) {
    return ABI ? (size_t)site * 12 + c : (size_t)c * V + site;
}

// Phase 1: thread (s, h, c[, a]) of the CTA's sites leaves row(s) a of
// M (psi_up + s C psi_dn)_c of hop h in sx[((h * 2 + c) * 3 + a) * S + s].
// The coordinate of `site` along nu decides the neighbour; sites past V use V - 1.
// CG: read `in` past the L1 cache (vectors that the running kernel itself writes).
template <int S, int SPLIT, bool ABI, bool CG = false>
__device__ __forceinline__ void s64_hops(const double2* __restrict__ U, const double2* in, const Geom& g,
                                         int site0, double2* __restrict__ sx, int tid) {
    constexpr int ROWS = 3 / SPLIT;
    const int s = tid % S, hc = (tid / S) & 15, a0 = SPLIT == 1 ? 0 : tid / (16 * S);
    const int h = hc >> 1, c = hc & 1, nu = h >> 1;
    const bool fwd = (h & 1) != 0;
    const int V = g.V;
    const int site = min(site0 + s, V - 1);
    const int L = nu == 0 ? g.Lx : nu == 1 ? g.Ly : nu == 2 ? g.Lz : g.Lt;
    const int stride = nu == 0 ? 1 : nu == 1 ? g.Lx : nu == 2 ? g.Lx * g.Ly : g.Lx * g.Ly * g.Lz;
    const int x = (int)(((unsigned)site / (unsigned)stride) % (unsigned)L);
    const int sn = fwd ? (x == L - 1 ? site - (L - 1) * stride : site + stride)
                       : (x == 0 ? site + (L - 1) * stride : site - stride);
    // M = U(x - nu) backward, U(x)^dagger forward: row a, column b
    const double2* __restrict__ Ul = U + (size_t)(nu * 9) * V + (fwd ? site : sn);
    const int ra = fwd ? 1 : 3, rb = fwd ? 3 : 1;
    const unsigned mc = fwd ? 0x80000000u : 0u;
    double2 m[ROWS][3], up[3], dn[3];
    // (C_nu psi_dn)_c = i^q psi_ic: nu = x: i^3 psi_3, i^3 psi_2; y: i^2 psi_3, psi_2;
    // z: i^3 psi_2, i psi_3; t: psi_2, psi_3; forward hops take the opposite sign (q + 2)
    const int ic = nu < 2 ? 3 - c : 2 + c;
    const int q = (nu == 0 ? 3 : nu == 1 ? (c ? 0 : 2) : nu == 2 ? (c ? 1 : 3) : 0) + (fwd ? 2 : 0);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const double2 *pu = in + comp_at<ABI>(3 * c + b, sn, V), *pd = in + comp_at<ABI>(3 * ic + b, sn, V);
        up[b] = CG ? __ldcg(pu) : *pu;
        dn[b] = CG ? __ldcg(pd) : *pd;
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
        for (int b = 0; b < 3; ++b) m[r][b] = Ul[(size_t)((a0 + r) * ra + b * rb) * V];
    double2 hh[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const double2 d = rot(dn[b], q);
        hh[b] = make_double2(up[b].x + d.x, up[b].y + d.y);
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        double2 v = make_double2(0.0, 0.0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double ex = m[r][b].x, ey = flip(m[r][b].y, mc), ny = flip(ey, 0x80000000u);
            v.x = fma(ny, hh[b].y, b == 0 ? ex * hh[b].x : fma(ex, hh[b].x, v.x));
            v.y = fma(ey, hh[b].x, b == 0 ? ex * hh[b].y : fma(ex, hh[b].y, v.y));
        }
        sx[((h * 2 + c) * 3 + a0 + r) * S + s] = v;
    }
}

// Phase 2: the sum over the eight hops for spin sp, colour a of slot s.
// (B_nu m)_0,1 of the lower spins: x: i m_1, i m_0; y: m_1, -m_0; z: i m_0,
// -i m_1; t: m_0, m_1, times -1 for the forward hops; wp_t, wm_t are the
// temporal weights of this site (with the boundary sign).
template <int S>
__device__ __forceinline__ double2 s64_sum(const double2* __restrict__ sx, int s, int sp, int a, double wp_t,
                                           double wm_t) {
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int h = 0; h < 8; ++h) {
        const int nu = h >> 1;
        const bool fwd = (h & 1) != 0;
        // column and i^q of spins 2 and 3
        const int col2 = nu < 2 ? 1 : 0, q2 = nu == 0 || nu == 2 ? 1 : 0;
        const int q3 = nu == 0 ? 1 : nu == 1 ? 2 : nu == 2 ? 3 : 0;
        const int col = sp < 2 ? sp : sp == 2 ? col2 : 1 - col2;
        const int q = sp < 2 ? 0 : (sp == 2 ? q2 : q3) + (fwd ? 2 : 0);
        const double2 b = rot(sx[((h * 2 + col) * 3 + a) * S + s], q);
        if (nu == 3) {
            const double w = fwd ? wm_t : wp_t;
            acc.x = fma(w, b.x, acc.x);
            acc.y = fma(w, b.y, acc.y);
        } else if (h == 0) {
            acc = b;
        } else {
            acc.x += b.x;
            acc.y += b.y;
        }
    }
    return acc;
}

// The temporal weights of a site: A uses (e^{mu}, e^{-mu}), A^dagger exchanges
// them; a hop across the antiperiodic t boundary carries -1.
__device__ __forceinline__ void t_weights(const Geom& g, int site, int dag, double emu, double emu_inv, double& wp,
                                          double& wm) {
    const int t = site / (g.Lx * g.Ly * g.Lz);
    wp = dag ? emu_inv : emu;
    wm = dag ? emu : emu_inv;
    if (g.antiperiodic && t == 0) wp = flip(wp, 0x80000000u);
    if (g.antiperiodic && t == g.Lt - 1) wm = flip(wm, 0x80000000u);
}

// ---- the stencil alone ------------------------------------------------------------
// One CTA per block of S sites and vector, the vector index fastest (the links
// of a block of sites come from HBM once and then from L2).
template <int S, bool ABI>
__global__ void __launch_bounds__(16 * S) k_stencil64(const double2* __restrict__ U, Geom g, DslashSet s0, DslashSet s1,
                                                      double kappa, double emu, double emu_inv) {
    __shared__ double2 sx[48 * S];
    pdl_trigger();
    pdl_wait();
    const int nvec = s0.n + s1.n;
    const int vec = blockIdx.x % nvec, site0 = (blockIdx.x / nvec) * S;
    const DslashSet& D = vec < s0.n ? s0 : s1;
    const int vi = vec < s0.n ? vec : vec - s0.n;
    const double2* in = reinterpret_cast<const double2*>(D.in) + (size_t)vi * D.in_stride;   // ordinary loads (nk_common.cuh)
    s64_hops<S, 1, ABI>(U, in, g, site0, sx, threadIdx.x);
    // component-fastest threads in the ABI layout, site-fastest in the device one (coalesced
    // stores).  12 of 16 threads sum: which warps idle rotates with the block of sites, as
    // the FP64 pipe of an SM sub-partition serves the warps of one residue mod 4
    const int tid = (threadIdx.x + 32 * ((blockIdx.x / nvec) & 3)) % (16 * S);
    const int s = ABI ? tid / 12 : tid % S, comp = ABI ? tid % 12 : tid / S;
    const int site = site0 + s;
    const bool live = tid < 12 * S && site < g.V;
    double2 p = make_double2(0.0, 0.0);
    if (live) p = in[comp_at<ABI>(comp, site, g.V)];
    __syncthreads();
    if (!live) return;
    double wp, wm;
    t_weights(g, site, D.dag, emu, emu_inv, wp, wm);
    const int sp = comp / 3;
    const double2 acc = s64_sum<S>(sx, s, sp, comp % 3, wp, wm);
    const unsigned sg = sp < 2 ? 0u : 0x80000000u;   // gamma5 = diag(1, 1, -1, -1)
    double2* __restrict__ out = D.out + (size_t)vi * D.out_stride;
    out[comp_at<ABI>(comp, site, g.V)] = make_double2(flip(fma(-kappa, acc.x, p.x), sg), flip(fma(-kappa, acc.y, p.y), sg));
}

__device__ __forceinline__ double2 caxpy_neg(double2 s, double2 c, double2 p) {   // s - c p
    return make_double2(fma(-c.x, p.x, fma(c.y, p.y, s.x)), fma(-c.x, p.y, fma(-c.y, p.x, s.y)));
}
__device__ __forceinline__ double2 caxpy_pos(double2 s, double2 c, double2 p) {   // s + c p
    return make_double2(fma(c.x, p.x, fma(-c.y, p.y, s.x)), fma(c.x, p.y, fma(c.y, p.x, s.y)));
}

// ---- fused with the first half of outer step j --------------------------------------
// (lanczos.cu describes the unnormalised basis q_j, p_j)
//   side 0: r = (A q_j) / n_j - (c_{j-1}/n_{j-1}) q_{j-1} -> q_{j+1},
//           H(j,j) = (p_j^dag r) / m_j^*  (Hermitian: Re(q_j^dag r) / n_j),
//   side 1: l = (A^dag p_j) / m_j - (beta^*_{j-1}/m_{j-1}) p_{j-1} -> p_{j+1}.
// The scalars of the step come from o.sc; the CTA that finishes last forms
// H(j,j) and the step-2 scalars.  CTA b of a vector walks a contiguous range
// of the site blocks; the grid is at most one wave (stencil64_blocks).
// In double-pass mode side 0 also accumulates y += c'_j q_j at its own site.
template <int S, int SPLIT, bool TS, bool PASS2>
__global__ void __launch_bounds__(16 * S * SPLIT, SPLIT == 1 ? kS64Sites / S : 1) k_stencil64_step1(const double2* __restrict__ U, Geom g, Outer o, int j,
                                                                    double kappa, double emu, double emu_inv, int nblk) {
    __shared__ double2 sx[48 * S];
    __shared__ double2 sh[33];
    const int nvec = TS ? 2 * o.n_rhs : o.n_rhs;
    const int vec = o.st_order == 0 ? blockIdx.x % nvec : blockIdx.x / nblk;
    const int blk = o.st_order == 0 ? blockIdx.x / nvec : blockIdx.x % nblk;
    const int side = vec / o.n_rhs;      // 0: A q_j, 1: A^dagger p_j
    const int rhs = vec % o.n_rhs;
    if (o.status[rhs] != kStatusOK) return;
    if (side == 1 && j == o.k - 1) return;   // the last step needs no left vector
    const double2* __restrict__ sc = o.sc + (size_t)rhs * kScalars;
    const double2 scl = sc[side ? kScM : kScN];     // 1/n_j (1/m_j)
    const double2 c1 = sc[side ? kScC1L : kScC1];   // zero at j = 0 (the previous vector is then any valid one)
    const int V = g.V, nsb = (V + S - 1) / S;
    const int b_lo = (int)((long)blk * nsb / nblk), b_hi = (int)((long)(blk + 1) * nsb / nblk);
    const int jp = j > 0 ? j - 1 : j;
    const double2* __restrict__ in = side ? outer_p(o, rhs, j) : outer_q(o, rhs, j);
    const double2* __restrict__ prv = side ? outer_p(o, rhs, jp) : outer_q(o, rhs, jp);
    double2* __restrict__ nxt = side ? outer_p(o, rhs, j + 1) : outer_q(o, rhs, j + 1);   // a scratch column at j = k - 1
    const double2* __restrict__ dotv = TS ? outer_p(o, rhs, j) : outer_q(o, rhs, j);
    double2* __restrict__ yacc = PASS2 ? o.y + (size_t)rhs * o.N : nullptr;
    const double2 cpj = PASS2 ? o.cp[(size_t)rhs * o.k + j] : make_double2(0.0, 0.0);
    const int tid = threadIdx.x;
    const int t2 = (tid + 32 * (blk & 3)) % (16 * S * SPLIT);   // idle warps rotate, as in k_stencil64
    const int s = t2 % S, comp = t2 / S, sp = comp / 3, a = comp % 3;
    const unsigned sg = sp < 2 ? 0u : 0x80000000u;   // gamma5 = diag(1, 1, -1, -1)
    double2 dot = make_double2(0.0, 0.0);
    for (int b = b_lo; b < b_hi; ++b) {
        s64_hops<S, SPLIT, false>(U, in, g, b * S, sx, threadIdx.x);
        const int site = b * S + s;
        const bool live = comp < 12 && site < V;
        const size_t idx = (size_t)comp * V + site;
        double2 p = make_double2(0.0, 0.0), pv = p, d = p;
        if (live) {
            p = in[idx];
            pv = prv[idx];
            if (side == 0) d = dotv[idx];
        }
        __syncthreads();
        if (live) {
            double wp, wm;
            t_weights(g, site, side, emu, emu_inv, wp, wm);
            const double2 acc = s64_sum<S>(sx, s, sp, a, wp, wm);
            const double2 v = make_double2(flip(fma(-kappa, acc.x, p.x), sg), flip(fma(-kappa, acc.y, p.y), sg));
            double2 rr;
            if (TS) {
                rr = caxpy_neg(cmul_fma(v, scl), c1, pv);
            } else {
                rr = make_double2(v.x * scl.x, v.y * scl.x);
                rr = make_double2(fma(-c1.x, pv.x, rr.x), fma(-c1.x, pv.y, rr.y));
            }
            nxt[idx] = rr;
            if (side == 0) {
                dot.x = fma(d.x, rr.x, fma(d.y, rr.y, dot.x));      // conj(d) r
                if (TS) dot.y = fma(d.x, rr.y, fma(-d.y, rr.x, dot.y));
                if (PASS2) yacc[idx] = caxpy_pos(yacc[idx], cpj, TS ? p : d);
            }
        }
        if (b + 1 < b_hi) __syncthreads();   // sx is rewritten
    }
    if (side != 0) return;
    const double2 part = block_sum(dot, sh);
    if (finish_partial(part, o.partials + (size_t)rhs * o.npart, o.counters + rhs, blk, nblk)) {
        const double2 tot = sum_partials(o.partials + (size_t)rhs * o.npart, nblk, sh);
        // Hermitian: H(j,j) = Re(q_j^dag r) / n_j, real (App. C); two-sided: (p_j^dag r) / m_j^*;
        // the step-2 scalars H(j,j)/n_j (warp 1) and H(j,j)^*/m_j (warp 0) side by side
        if (tid == 0 || tid == 32) {
            const double2 al = TS ? cmul_fma(sc[kScD], tot) : make_double2(tot.x * sc[kScD].x, 0.0);
            if (tid == 0) {
                o.alpha[(size_t)rhs * o.k + j] = al;
                o.counters[rhs] = 0u;
                o.sc[(size_t)rhs * kScalars + kScC4] = TS ? cmul_fma(cconj(al), sc[kScM]) : make_double2(0.0, 0.0);
            } else {
                o.sc[(size_t)rhs * kScalars + kScC3] = cmul_fma(al, sc[kScN]);
            }
        }
    }
}

// ---- a run of outer steps in one launch ----------------------------------------------
// Steps [j_lo, j_hi) of an FP64 recurrence.  A step of a small lattice is two
// kernels of 5 to 15 us whose launches, cold starts and one-CTA tails (partial
// sums, beta, gamma and the scalars on one lane, then a kernel boundary before
// anyone may use them) are half of it.  Here the CTAs stay: one cooperative
// launch, at most one CTA per SM and RHS share, and per step two grid barriers
// of the RHS's CTAs; after each every CTA adds the partial sums and forms the
// scalars for itself (the same values in the same order everywhere), so nothing
// waits for a second hop through memory.  128 (64) threads work on eight (four) sites as in
// k_stencil64_step1 (group of the CTA with its own named barrier), then all on
// (component pair, site) items as in k_step2.  Vectors written by the launch are
// read past L1.
// The barriers' waits are bounded: a CTA whose wait runs out marks its RHS
// kStatusTimeout and leaves; the others' waits then run out too.
// Measured, us per step against the step kernels: 4^4, mu = 0 13.5 -> 9.7; 6^4, mu = 0.1
// 21.0 -> 17.1; 10^4, mu = 0.2 58.1 -> 52.7 (all one source).  Registers capped for two
// CTAs per SM cost 4% at 10^4 (62.7 -> 65.2 ms a solve of k = 1024); 256 threads per CTA 18.5
// at 6^4, 55.5 at 10^4.
constexpr int kRunThreads = 384;
template <int S> constexpr int kRunGroup = 16 * S;                            // threads of a group on S sites
template <int S> constexpr int kRunGroups = kRunThreads / kRunGroup<S>;   // groups of a CTA

__device__ __forceinline__ unsigned long long run_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// All CTAs of one RHS (n of them; the counter counts arrivals since the launch).
// False if it waited for wait_ns.
__device__ __forceinline__ bool run_barrier(unsigned* counter, unsigned target, unsigned long long wait_ns, bool* ok_sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
        bool ok = true;
        if (ld_acquire(counter) < target) {
            const unsigned long long t0 = run_ns();
            while (ld_acquire(counter) < target)
                if (run_ns() - t0 >= wait_ns) { ok = false; break; }
        }
        *ok_sh = ok;
    }
    __syncthreads();
    return *ok_sh;
}

// What the two forms of a run share.  Every CTA of an RHS (`ncta` of them) holds the
// step's scalars in sc; part1 and part2 are its partial sums of H(j,j) and of delta.
// The sums below have one order whatever the form, and products of complex
// scalars are written as explicit fused multiply-adds, so that both forms give
// the same bits.

// Sum of the ncta partials in every lane of one warp.
__device__ __forceinline__ double2 run_total(const double2* part, int ncta) {
    const int lane = threadIdx.x % 32;
    double2 a = make_double2(0.0, 0.0);
    for (int i = lane; i < ncta; i += 32) {
        const double2 v = __ldcg(part + i);
        a = i == lane ? v : cadd(a, v);
    }
    const double t = warp_sum_split(a);
    return make_double2(__shfl_sync(0xffffffffu, t, 0), __shfl_sync(0xffffffffu, t, 16));
}

// First half of step j, stencil and step 1 on this CTA's share of the site blocks;
// returns the thread's part of H(j,j).
template <bool TS, bool PASS2, int S>
__device__ __forceinline__ double2 run_half1(const double2* __restrict__ U, const Geom& g, const Outer& o, int rhs, int j,
                                             int cta, int ncta, const double2* sc, double2 (*sx)[48 * S],
                                             double kappa, double emu, double emu_inv) {
    const int tid = threadIdx.x, grp = tid / kRunGroup<S>, gt = tid % kRunGroup<S>;
    const int V = g.V, nsb = (V + S - 1) / S;
    const int jp = j > 0 ? j - 1 : j;
    const bool left = TS && j < o.k - 1;
    // the warp that idles in the sum differs from group to group (FP64 pipes, as in k_stencil64)
    const int t2 = (gt + 32 * (grp & 3)) % kRunGroup<S>;
    const int s = t2 % S, comp = t2 / S, sp = comp / 3, a = comp % 3;
    const unsigned sg = sp < 2 ? 0u : 0x80000000u;
    double2 dot = make_double2(0.0, 0.0);
    for (int u = cta + ncta * grp; u < (left ? 2 : 1) * nsb; u += ncta * kRunGroups<S>) {
        const int side = u >= nsb ? 1 : 0, b = u - side * nsb;
        const double2* in = side ? outer_p(o, rhs, j) : outer_q(o, rhs, j);
        s64_hops<S, 1, false, true>(U, in, g, b * S, sx[grp], gt);
        const int site = b * S + s;
        const bool live = comp < 12 && site < V;
        const size_t idx = (size_t)comp * V + site;
        double2 p = make_double2(0.0, 0.0), pv = p, d = p;
        if (live) {
            p = __ldcg(in + idx);
            pv = __ldcg((side ? outer_p(o, rhs, jp) : outer_q(o, rhs, jp)) + idx);
            if (side == 0) d = __ldcg((TS ? outer_p(o, rhs, j) : outer_q(o, rhs, j)) + idx);
        }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(kRunGroup<S>) : "memory");
        if (live) {
            double wp, wm;
            t_weights(g, site, side, emu, emu_inv, wp, wm);
            const double2 acc = s64_sum<S>(sx[grp], s, sp, a, wp, wm);
            const double2 v = make_double2(flip(fma(-kappa, acc.x, p.x), sg), flip(fma(-kappa, acc.y, p.y), sg));
            const double2 scl = sc[side ? kScM : kScN], c1 = sc[side ? kScC1L : kScC1];
            double2 rr;
            if (TS) {
                rr = caxpy_neg(cmul_fma(v, scl), c1, pv);
            } else {
                rr = make_double2(v.x * scl.x, v.y * scl.x);
                rr = make_double2(fma(-c1.x, pv.x, rr.x), fma(-c1.x, pv.y, rr.y));
            }
            (side ? outer_p(o, rhs, j + 1) : outer_q(o, rhs, j + 1))[idx] = rr;
            if (side == 0) {
                dot.x = fma(d.x, rr.x, fma(d.y, rr.y, dot.x));      // conj(d) r
                if (TS) dot.y = fma(d.x, rr.y, fma(-d.y, rr.x, dot.y));
                if (PASS2) {
                    double2* y = o.y + (size_t)rhs * o.N + idx;
                    *y = caxpy_pos(*y, o.cp[(size_t)rhs * o.k + j], TS ? p : d);
                }
            }
        }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(kRunGroup<S>) : "memory");   // sx is rewritten
    }
    return dot;
}

// H(j,j) and the step-2 scalars, by one warp (an FP64 warp instruction costs its
// pipe as much as any).  Hermitian: H(j,j) = Re(q_j^dag r) / n_j, real (App. C);
// two-sided: (p_j^dag r) / m_j^*.
template <bool TS>
__device__ __forceinline__ void run_alpha(const Outer& o, int rhs, int j, bool write, int ncta, const double2* part1, double2* sc) {
    const double2 tot = run_total(part1, ncta);
    const double2 al = TS ? cmul_fma(sc[kScD], tot) : make_double2(tot.x * sc[kScD].x, 0.0);
    if (threadIdx.x % 32 == 0) {
        if (write) o.alpha[(size_t)rhs * o.k + j] = al;
        sc[kScC3] = cmul_fma(al, sc[kScN]);
        sc[kScC4] = TS ? cmul_fma(cconj(al), sc[kScM]) : make_double2(0.0, 0.0);
    }
}

// Second half of step j on this CTA's share of the (component pair, site) items;
// returns the thread's part of delta.
template <bool TS>
__device__ __forceinline__ double2 run_half2(const Outer& o, int rhs, int j, int cta, int ncta, const double2* sc) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const unsigned V = (unsigned)(o.N / 12), items = 6u * V;
    const double2 c3 = sc[kScC3], c4 = sc[kScC4];
    const double2* qj = outer_q(o, rhs, j);
    double2* r = outer_q(o, rhs, j + 1);
    const double2* pj = TS ? outer_p(o, rhs, j) : nullptr;
    double2* l = TS ? outer_p(o, rhs, j + 1) : nullptr;
    double2 del = make_double2(0.0, 0.0);
    const unsigned stride = (unsigned)ncta * kRunThreads;
    for (unsigned i = (unsigned)(cta + ncta * warp) * 32u + lane; i < items; i += stride) {
        const size_t e0 = (size_t)i + (size_t)(i / V) * V;   // component 2 cp of the item
        double2 q[2], x[2], pv[2], w[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const size_t e = e0 + (size_t)h * V;
            q[h] = __ldcg(qj + e);
            x[h] = __ldcg(r + e);
            if (TS) { pv[h] = __ldcg(pj + e); w[h] = __ldcg(l + e); }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const size_t e = e0 + (size_t)h * V;
            x[h] = TS ? caxpy_neg(x[h], c3, q[h])
                      : make_double2(fma(-c3.x, q[h].x, x[h].x), fma(-c3.x, q[h].y, x[h].y));
            r[e] = x[h];
            if (TS) {
                w[h] = caxpy_neg(w[h], c4, pv[h]);
                l[e] = w[h];
                del.x = fma(x[h].x, w[h].x, fma(x[h].y, w[h].y, del.x));   // conj(r) l
                del.y = fma(x[h].x, w[h].y, fma(-x[h].y, w[h].x, del.y));
            } else {
                del.x = fma(x[h].x, x[h].x, fma(x[h].y, x[h].y, del.x));
            }
        }
    }
    return del;
}

// beta_j, gamma_j and the scalars of step j + 1, by one warp; *go: no breakdown.
template <bool TS>
__device__ __forceinline__ void run_beta(const Outer& o, int rhs, int j, bool write, int ncta, const double2* part2, double2* sc,
                                         bool* go) {
    const StepScalars t = step_scalars<TS>(run_total(part2, ncta));
    if (threadIdx.x % 32 == 0) {
        if (write) {
            o.beta[(size_t)rhs * o.k + j] = t.beta;
            o.gamma[(size_t)rhs * o.k + j] = t.gamma;
            if (!t.ok) mark_failed(o, rhs, kStatusBreakdown);
        }
        *go = t.ok;
        if (t.ok) next_scalars<TS>(sc, t);
    }
}

template <bool TS, bool PASS2, int S>
__global__ void __launch_bounds__(kRunThreads) k_run64(const double2* __restrict__ U, Geom g, Outer o, int j_lo, int j_hi,
                                                          double kappa, double emu, double emu_inv,
                                                          unsigned long long wait_ns) {
    __shared__ double2 sx[kRunGroups<S>][48 * S];
    __shared__ double2 sh[33];
    __shared__ double2 sc[kScalars];
    __shared__ bool ok_sh;   // a barrier's outcome (written inside run_barrier only)
    __shared__ bool go_sh;   // no breakdown at this step
    const int rhs = blockIdx.x % o.n_rhs, cta = blockIdx.x / o.n_rhs, ncta = gridDim.x / o.n_rhs;
    if (o.status[rhs] != kStatusOK) return;
    const int tid = threadIdx.x;
    unsigned* counter = o.run_bar + rhs;
    unsigned target = 0;
    double2* part1 = o.partials + (size_t)rhs * o.npart;
    double2* part2 = part1 + ncta;
    if (tid < kScalars) sc[tid] = o.sc[(size_t)rhs * kScalars + tid];
    __syncthreads();
    for (int j = j_lo; j < j_hi; ++j) {
        const double2 dot = block_sum(run_half1<TS, PASS2, S>(U, g, o, rhs, j, cta, ncta, sc, sx, kappa, emu, emu_inv), sh);
        if (tid == 0) part1[cta] = dot;
        target += (unsigned)ncta;
        if (!run_barrier(counter, target, wait_ns, &ok_sh)) {
            if (tid == 0) mark_failed(o, rhs, kStatusTimeout);
            return;
        }
        if (tid < 32) run_alpha<TS>(o, rhs, j, cta == 0, ncta, part1, sc);
        __syncthreads();
        if (j == o.k - 1) break;
        const double2 del = block_sum(run_half2<TS>(o, rhs, j, cta, ncta, sc), sh);
        if (tid == 0) part2[cta] = del;
        target += (unsigned)ncta;
        if (!run_barrier(counter, target, wait_ns, &ok_sh)) {
            if (tid == 0) mark_failed(o, rhs, kStatusTimeout);
            return;
        }
        if (tid < 32) run_beta<TS>(o, rhs, j, cta == 0, ncta, part2, sc, &go_sh);
        __syncthreads();
        if (!go_sh) return;   // the same decision in every CTA of the RHS
    }
    if (cta == 0 && tid < kScalars && j_hi < o.k) o.sc[(size_t)rhs * kScalars + tid] = sc[tid];
}

// The same steps with a launch in the place of each grid barrier, for solves that
// share the chip with others: the CTAs of k_run64 hold their SMs from the first
// step to the last, and a second solve waits for a place; these come and go.  HALF 0
// is the first half of step j, HALF 1 the second; the CTA that finishes last forms
// the scalars, for all (formed by every CTA, as in k_run64, they would take an SM's
// FP64 pipe from the other solves: 10.4 against 8.4 below).  us per step of one of 16
// solves in flight, all steps in one launch -> a launch per half step: 4^4, mu = 0.1 3.4 -> 3.1;
// 6^4, mu = 0.1 11.2 -> 8.4; 8^4 21.8 -> 18.3; 10^4, mu = 0.2 46.2 -> 40.2 (k_run64 there with
// registers for three CTAs per SM; one per SM 14 at 6^4); of one alone 12.7 -> 17.3, 17.1 -> 22.6,
// 27.9 -> 33.7, 52.7 -> 59.4.
template <bool TS, bool PASS2, int HALF, int S>
__global__ void __launch_bounds__(kRunThreads, HALF == 0 ? 2 : 3) k_run64_half(const double2* __restrict__ U, Geom g, Outer o, int j,
                                                               double kappa, double emu, double emu_inv) {
    __shared__ double2 sx[HALF == 0 ? kRunGroups<S> : 1][48 * S];
    __shared__ double2 sh[33];
    __shared__ double2 sc[kScalars];
    __shared__ bool go_sh;
    const int rhs = blockIdx.x % o.n_rhs, cta = blockIdx.x / o.n_rhs, ncta = gridDim.x / o.n_rhs;
    if (o.status[rhs] != kStatusOK) return;
    const int tid = threadIdx.x;
    double2* part = o.partials + (size_t)rhs * o.npart;
    double2* home = o.sc + (size_t)rhs * kScalars;
    if (tid < kScalars) sc[tid] = home[tid];
    __syncthreads();
    const double2 mine = HALF == 0 ? run_half1<TS, PASS2, S>(U, g, o, rhs, j, cta, ncta, sc, sx, kappa, emu, emu_inv)
                                   : run_half2<TS>(o, rhs, j, cta, ncta, sc);
    if (!finish_partial(block_sum(mine, sh), part, o.counters + rhs, cta, ncta)) return;
    __threadfence();
    if (tid < 32) {
        if (HALF == 0) run_alpha<TS>(o, rhs, j, true, ncta, part, sc);
        else run_beta<TS>(o, rhs, j, true, ncta, part, sc, &go_sh);
    }
    __syncthreads();
    if (tid < kScalars) home[tid] = sc[tid];   // every other CTA has read its copy
    if (tid == 0) o.counters[rhs] = 0u;
}

// Sites of a group and CTAs per RHS of a run.  One CTA per SM over the RHS, fewer where
// there are not so many blocks of eight sites.  Eight sites per group waste no lanes
// in the sum over the hops; with one to three blocks of eight per CTA, groups of four
// share them out more evenly (us per step, four / eight: 6^4 1 vector 11.5 / 12.0, 2 vectors
// 17.1 / 17.7, 5x4x3x6 x 2 x 2 13.8 / 14.4; one block or less: 4^4 1 9.9 / 9.6, 2 13.5 / 12.7; more
// than three: 8^4 1 17.9 / 17.3, 2 29.5 / 28.0, 10^4 2 54.4 / 52.7).
struct RunShape {
    int sites, ctas;
};
RunShape run_shape(const Geom& g, const Outer& o, int sms) {
    const int most = std::max(1, sms / o.n_rhs), blocks = (o.two_sided ? 2 : 1) * ((g.V + 7) / 8);
    return {blocks > most && blocks <= 3 * most ? 4 : 8, std::min(most, blocks)};
}

template <int S, int SPLIT>
void launch_s64_step1(const double2* U, const Geom& g, const Outer& o, int j, double kappa, double emu, double emu_inv,
                      cudaStream_t st) {
    const int nvec = o.two_sided ? 2 * o.n_rhs : o.n_rhs;
    const int nblk = stencil64_blocks(g, 16 * S, nvec);
    const unsigned grid = (unsigned)nblk * (unsigned)nvec;
    constexpr int T = 16 * S * SPLIT;
    const bool pass2 = o.y != nullptr;
    if (o.two_sided) {
        if (pass2) k_stencil64_step1<S, SPLIT, true, true><<<grid, T, 0, st>>>(U, g, o, j, kappa, emu, emu_inv, nblk);
        else k_stencil64_step1<S, SPLIT, true, false><<<grid, T, 0, st>>>(U, g, o, j, kappa, emu, emu_inv, nblk);
    } else {
        if (pass2) k_stencil64_step1<S, SPLIT, false, true><<<grid, T, 0, st>>>(U, g, o, j, kappa, emu, emu_inv, nblk);
        else k_stencil64_step1<S, SPLIT, false, false><<<grid, T, 0, st>>>(U, g, o, j, kappa, emu, emu_inv, nblk);
    }
}

}  // namespace

// CTAs (and partial sums) per vector of the fused kernel with `threads`
// threads per CTA at split 1 (threads / 16 sites): one per block of sites, but
// no more than one wave of the chip over all vectors
int stencil64_blocks(const Geom& g, int threads, int nvec) {
    const int S = threads / 16;
    const int nsb = (g.V + S - 1) / S;
    const int wave = device_sms() * (kS64Sites / S) / nvec;
    return nsb < wave ? nsb : (wave > 0 ? wave : 1);
}

void launch_stencil64_step1(const void* U64, const Geom& g, const Outer& o, int j, double kappa, double mu,
                            cudaStream_t st) {
    const double2* U = (const double2*)U64;
    const double ep = exp(mu), em = exp(-mu);
#define NK_S64(S_)                                                                    \
    do {                                                                              \
        if (o.st_split == 3) launch_s64_step1<S_, 3>(U, g, o, j, kappa, ep, em, st);  \
        else launch_s64_step1<S_, 1>(U, g, o, j, kappa, ep, em, st);                  \
    } while (0)
    if (o.st_threads == 64) NK_S64(4);
    else if (o.st_threads == 128) NK_S64(8);
    else NK_S64(16);
#undef NK_S64
}

bool launch_run64(const void* U64, const Geom& g, const Outer& o, int j_lo, int j_hi, double kappa, double mu, int sms,
                  unsigned long long wait_ns, cudaStream_t st) {
    cudaMemsetAsync(o.run_bar, 0, sizeof(unsigned) * o.n_rhs, st);
    cudaLaunchConfig_t cfg = {};
    const RunShape sh = run_shape(g, o, sms);
    cfg.gridDim = dim3((unsigned)(sh.ctas * o.n_rhs));
    cfg.blockDim = dim3(kRunThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const double2* U = (const double2*)U64;
    const double ep = exp(mu), em = exp(-mu);
    const bool pass2 = o.y != nullptr;
#define NK_RUN(TS_, P2_)                                                                                            \
    (sh.sites == 4 ? cudaLaunchKernelEx(&cfg, k_run64<TS_, P2_, 4>, U, g, o, j_lo, j_hi, kappa, ep, em, wait_ns) \
                   : cudaLaunchKernelEx(&cfg, k_run64<TS_, P2_, 8>, U, g, o, j_lo, j_hi, kappa, ep, em, wait_ns))
    const cudaError_t e = o.two_sided ? (pass2 ? NK_RUN(true, true) : NK_RUN(true, false))
                                      : (pass2 ? NK_RUN(false, true) : NK_RUN(false, false));
#undef NK_RUN
    return e == cudaSuccess;
}

void launch_run64_half(const void* U64, const Geom& g, const Outer& o, int half, int j, double kappa, double mu, int sms,
                       cudaStream_t st) {
    const RunShape sh = run_shape(g, o, sms);
    const unsigned grid = (unsigned)(sh.ctas * o.n_rhs);
    const double ep = exp(mu), em = exp(-mu);
#define NK_HALF(TS_, P2_, H_, S_) k_run64_half<TS_, P2_, H_, S_><<<grid, kRunThreads, 0, st>>>((const double2*)U64, g, o, j, kappa, ep, em)
#define NK_HALF0(TS_, P2_)                           \
    do {                                              \
        if (sh.sites == 4) NK_HALF(TS_, P2_, 0, 4);   \
        else NK_HALF(TS_, P2_, 0, 8);                 \
    } while (0)
    if (half == 0) {
        if (o.two_sided) { if (o.y) NK_HALF0(true, true); else NK_HALF0(true, false); }
        else { if (o.y) NK_HALF0(false, true); else NK_HALF0(false, false); }
    } else {   // (does not see the sites)
        if (o.two_sided) NK_HALF(true, false, 1, 8); else NK_HALF(false, false, 1, 8);
    }
#undef NK_HALF0
#undef NK_HALF
}

void launch_stencil64(const void* U64, const Geom& g, const DslashSet& s0, const DslashSet& s1, bool abi, double kappa,
                      double mu, cudaStream_t st) {
    const int nvec = s0.n + s1.n;
    if (nvec == 0) return;
    constexpr int S = 8;
    const unsigned grid = (unsigned)((g.V + S - 1) / S) * (unsigned)nvec;
    if (abi) launch_kernel(k_stencil64<S, true>, grid, 16 * S, 0, st, true, (const double2*)U64, g, s0, s1, kappa, exp(mu), exp(-mu));
    else launch_kernel(k_stencil64<S, false>, grid, 16 * S, 0, st, true, (const double2*)U64, g, s0, s1, kappa, exp(mu), exp(-mu));
}

}  // namespace nk

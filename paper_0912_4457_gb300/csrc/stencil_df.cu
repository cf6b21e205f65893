// Multi-RHS two-float (about 48-bit) Wilson stencil A = gamma5 D_w(mu),
// A^dagger = gamma5 D_w(-mu) (Sec. 2): the stencil of the early outer steps of
// the mixed schedule, where an FP32 stencil would cost accuracy the later
// steps cannot recover.
//
// One CTA owns a block of kDfSites consecutive sites for every vector of the
// launch (threadIdx.x = site in the block, threadIdx.y = vector, for few vectors
// two threads of one).  Before any
// vector is touched the CTA stages, in shared memory, the links of its sites'
// eight hops in the form the arithmetic uses -- M = U(x - nu) for the backward
// hops, M = U(x)^dagger for the forward ones, each element's real and
// imaginary part as broadcast pairs (hi, hi) and (lo, lo) -- with the
// neighbour indices and the boundary signs; every vector then reuses them.
//
// The arithmetic is two-float (a value is hi + lo, about 48 significant
// bits: TwoSum and TwoProd on the FP32 pipe) in the packed two-lane FP32
// instructions of sm_100+ (nk_f32x2.cuh): the two lanes carry the two
// half-spinor columns of a hop, which multiply the same link element, so one
// instruction serves both.  Per colour b a spinor is held as UR = (psi_0.re,
// psi_1.re), UI = (psi_0.im, psi_1.im), DR, DI (spins 2, 3).
//
// Input: two-float vectors (dfc, [vector][12][V]); output: FP64 vectors
// ([vector][12][V], or the ABI layout [vector][V][12]) of gamma5 (psi - kappa hops), optionally scaled by the
// step scalar 1/n_j (A) or 1/m_j (A^dagger) in two-float arithmetic -- the
// input of the FP64 step-1 kernel.
#include "nk_common.cuh"
#include "nk_f32x2.cuh"
#include "nk_kernels.h"

namespace nk {

namespace {

constexpr int kDfSites = 8;                        // sites per CTA
constexpr int kDfMaxThreads = kDfSites * 24;   // 12 RHS of A and 12 of A^dagger

struct DfSmem {
    ulonglong2* lk;   // [((h * 9 + e) * 2 + part) * kDfSites + s]: part 0 re, 1 im, as {(hi, hi), (lo, lo)}
    int* nb;          // [h * kDfSites + s]
    float* fl;        // [h * kDfSites + s]: -1 across the antiperiodic t boundary, else 1
};

constexpr size_t df_smem() { return (size_t)kDfSites * (8 * 9 * 2 * 16 + 8 * 4 + 8 * 4); }

__device__ __forceinline__ DfSmem df_carve(char* sm) {
    DfSmem r;
    r.lk = reinterpret_cast<ulonglong2*>(sm);
    r.nb = reinterpret_cast<int*>(sm + (size_t)kDfSites * 8 * 9 * 2 * 16);
    r.fl = reinterpret_cast<float*>(sm + (size_t)kDfSites * (8 * 9 * 2 * 16 + 8 * 4));
    return r;
}

// Neighbour indices, boundary signs and the hop matrices of the CTA's sites
// (hop h: nu = h / 2, odd h forward).  Sites past V use site V - 1.
__device__ __forceinline__ void df_stage(const dfc* __restrict__ U, const Geom& g, int site0, const DfSmem& S) {
    const int tx = threadIdx.x, ty = threadIdx.y, vg = blockDim.y;
    const int site = min(site0 + tx, g.V - 1);
    if (ty == 0) {
        const int L[4] = {g.Lx, g.Ly, g.Lz, g.Lt};
        const int stride[4] = {1, g.Lx, g.Lx * g.Ly, g.Lx * g.Ly * g.Lz};
        int c[4];
        int r = site;
#pragma unroll
        for (int d = 0; d < 4; ++d) { c[d] = r % L[d]; r /= L[d]; }
#pragma unroll
        for (int h = 0; h < 8; ++h) {
            const int nu = h >> 1;
            const bool fwd = (h & 1) != 0;
            const bool wrap = fwd ? c[nu] == L[nu] - 1 : c[nu] == 0;
            const int sn = fwd ? (wrap ? site - (L[nu] - 1) * stride[nu] : site + stride[nu])
                               : (wrap ? site + (L[nu] - 1) * stride[nu] : site - stride[nu]);
            S.nb[h * kDfSites + tx] = sn;
            S.fl[h * kDfSites + tx] = (nu == 3 && g.antiperiodic && wrap) ? -1.0f : 1.0f;
        }
    }
    __syncthreads();
#pragma unroll 2
    for (int q = ty; q < 72; q += vg) {   // (two elements in flight: few vectors make many rounds)
        const int h = q / 9, e = q % 9, nu = h >> 1, a = e / 3, b = e % 3;
        const bool fwd = (h & 1) != 0;
        // M_ab = U(x - nu)_ab backward, conj(U(x)_ba) forward
        const dfc u = fwd ? U[(size_t)(nu * 9 + 3 * b + a) * g.V + site]
                          : U[(size_t)(nu * 9 + e) * g.V + S.nb[h * kDfSites + tx]];
        const float ih = fwd ? -u.y.hi : u.y.hi, il = fwd ? -u.y.lo : u.y.lo;
        S.lk[(q * 2 + 0) * kDfSites + tx] = make_ulonglong2(pk(u.x.hi, u.x.hi), pk(u.x.lo, u.x.lo));
        S.lk[(q * 2 + 1) * kDfSites + tx] = make_ulonglong2(pk(ih, ih), pk(il, il));
    }
    __syncthreads();
}

struct DSpin {
    P2 ur[3], ui[3], dr[3], di[3];
};

// the two-float spinor of site s (components 3 sp + b, each (re.hi, re.lo,
// im.hi, im.lo)) in the spin-pair lanes; SWAP exchanges the lanes of the lower pair.
// Ordinary loads: the vectors may have been written while this grid was already alive
// (nk_common.cuh).
__device__ __forceinline__ void load_dspin(const dfc* in, int V, int s, DSpin& p, bool swap) {
    const float4* f = reinterpret_cast<const float4*>(in) + s;
    const float4* f2 = f + (size_t)(swap ? 9 : 6) * V;
    const float4* f3 = f + (size_t)(swap ? 6 : 9) * V;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const float4 s0 = ld_after_wait(f + (size_t)b * V), s1 = ld_after_wait(f + (size_t)(3 + b) * V);
        const float4 s2 = ld_after_wait(f2 + (size_t)b * V), s3 = ld_after_wait(f3 + (size_t)b * V);
        p.ur[b] = {pk(s0.x, s1.x), pk(s0.y, s1.y)};
        p.ui[b] = {pk(s0.z, s1.z), pk(s0.w, s1.w)};
        p.dr[b] = {pk(s2.x, s3.x), pk(s2.y, s3.y)};
        p.di[b] = {pk(s2.z, s3.z), pk(s2.w, s3.w)};
    }
}

// sign-bit masks of the two lanes
constexpr f2p kNeg0 = 0x0000000080000000ull, kNeg1 = 0x8000000000000000ull, kNeg = kNeg0 | kNeg1;
__device__ __forceinline__ P2 sgn(P2 a, f2p m) { return {a.s ^ m, a.e ^ m}; }

// One hop into the accumulators: acc += w (1 + s gamma_nu) M psi_n with
// s = +1 backward (M = U(x - nu)), -1 forward (M = U(x)^dagger), in the
// chiral basis:
//   (C psi_dn)_{0,1}:  nu = x: -i psi_3, -i psi_2;  y: -psi_3, psi_2;
//                      z: -i psi_2, i psi_3;       t: psi_2, psi_3
//   (B m)_{0,1}:       nu = x: i m_1, i m_0;        y: m_1, -m_0;
//                      z: i m_0, -i m_1;           t: m_0, m_1
// (i z = (-z.im, z.re)).  x and y exchange the two lower spins: their lower
// pair is loaded, and the accumulators' lower pair held, with the lanes
// swapped.  With that, x and z (EVEN) have the same form but for lane signs,
// and so have y and t: two instantiations for the eight hops, direction and
// sense as sign masks.  Instruction fetch is what this saves: eight unrolled
// hops overflowed the instruction cache, and with one instantiation per
// direction a warp still waited 0.7 of 6 cycles per instruction for it.
template <bool EVEN>
__device__ __forceinline__ void df_hop(DSpin& acc, const dfc* in, int V, const DfSmem& S, df wp_t,
                                       df wm_t, bool swap, int fwd) {
    const int H = 2 * ((swap ? 0 : 2) + (EVEN ? 0 : 1)) + fwd;
    const f2p m = fwd ? kNeg : 0ull;
    const f2p k = m ^ (EVEN ? (swap ? 0ull : kNeg1) : (swap ? kNeg0 : 0ull));
    const int tx = threadIdx.x;
    DSpin p;
    load_dspin(in, V, S.nb[H * kDfSites + tx], p, swap);
    // projection: HR = (h0.re, h1.re), HI = (h0.im, h1.im) per colour, and -HI
    P2 hr[3], hi[3], nhi[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (EVEN) {   // x: c = -i (psi3, psi2); z: c = -i (psi2, -psi3)
            hr[b] = p2_add(p.ur[b], sgn(p.di[b], k));
            hi[b] = p2_add(p.ui[b], sgn(p.dr[b], k ^ kNeg));
        } else {      // y: c = (-psi3, psi2); t: c = (psi2, psi3)
            hr[b] = p2_add(p.ur[b], sgn(p.dr[b], k));
            hi[b] = p2_add(p.ui[b], sgn(p.di[b], k));
        }
        nhi[b] = p2_neg(hi[b]);
    }
    const bool temporal = !EVEN && !swap;
    P2 wt = {0ull, 0ull};   // the temporal weight e^{+-mu} with the boundary sign (t hops only)
    if (temporal) {
        const df w = fwd ? wm_t : wp_t;
        const float f = S.fl[H * kDfSites + tx];
        wt = {pk(w.hi * f, w.hi * f), pk(w.lo * f, w.lo * f)};
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        P2 xr, xi;   // (x0, x1) = row a of M times (h0, h1)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int q = H * 9 + 3 * a + b;
            const ulonglong2 mr2 = S.lk[(q * 2 + 0) * kDfSites + tx], mi2 = S.lk[(q * 2 + 1) * kDfSites + tx];
            const P2 mr = {mr2.x, mr2.y}, mi = {mi2.x, mi2.y};
            if (b == 0) {
                xr = p2_prod(mr, hr[b]);
                xi = p2_prod(mr, hi[b]);
            } else {
                p2_add_prod(xr, mr, hr[b]);
                p2_add_prod(xi, mr, hi[b]);
            }
            p2_add_prod(xr, mi, nhi[b]);   // re: mr hr - mi hi
            p2_add_prod(xi, mi, hr[b]);    // im: mr hi + mi hr
        }
        if (!EVEN) {
            if (temporal) {
                xr = p2_prod(wt, xr);
                xi = p2_prod(wt, xi);
            }
        }
        acc.ur[a] = p2_add(acc.ur[a], xr);
        acc.ui[a] = p2_add(acc.ui[a], xi);
        if (EVEN) {   // lanes as accumulated, x: (b1, b0) = i (x0, x1); z: (b0, b1) = i (x0, -x1)
            acc.dr[a] = p2_add(acc.dr[a], sgn(xi, k ^ kNeg));
            acc.di[a] = p2_add(acc.di[a], sgn(xr, k));
        } else {      // y: (b1, b0) = (-x0, x1); t: (b0, b1) = (x0, x1)
            acc.dr[a] = p2_add(acc.dr[a], sgn(xr, k));
            acc.di[a] = p2_add(acc.di[a], sgn(xi, k));
        }
    }
}

// two lanes of a two-float pair as FP64 (integer-pipe conversions, one FP64 add)
__device__ __forceinline__ void p2_to_double(P2 v, double& l0, double& l1) {
    float s0, s1, e0, e1;
    upk(v.s, s0, s1);
    upk(v.e, e0, e1);
    l0 = f2d_int(s0) + f2d_int(e0);
    l1 = f2d_int(s1) + f2d_int(e1);
}

// the value of the lane 8 away, within the 16 lanes of one vector
__device__ __forceinline__ P2 shfl_half(P2 v) {
    const unsigned lanes = 0xffffu << (threadIdx.y & 2 ? 16 : 0);
    return {__shfl_xor_sync(lanes, (unsigned long long)v.s, 8), __shfl_xor_sync(lanes, (unsigned long long)v.e, 8)};
}

// SPLIT = 2: two threads share a site and vector, one takes the backward and one
// the forward hops, and each finishes one spin pair (24 words exchanged, 6 sums).
// Half the work a thread fills a launch of few vectors' lanes and halves its last
// wave; it costs the exchange and a CTA of twice the threads.  Measured, one
// application, 1 -> 2 threads: 10^4 sites, 1 vector 32.8 -> 20.0 us, 3 31.3 ->
// 27.0, 6 45.9 -> 37.1, 8 46.9 -> 44.4; 16^3 x 32, 1 461 -> 251, 6 500 -> 452.
// Where many waves hide the last one only the exchange is left: 8 at 16384 sites
// 67.3 -> 68.7, at 131072 506 -> 528; 12 at 8^4 inside a step 31 -> 33.
// At 9 to 12 vectors a CTA of one thread each is three warps, which fill the four
// schedulers unevenly: there two threads win once many waves follow one another
// (12 vectors: 228 -> 208 us at 32768, 455 -> 409 at 65536; a step of
// 12^4, 6 two-sided sources, 209 -> 202), and not before (10^4, 12 sources 98 -> 100).
constexpr int kDfSplit = 6;            // vectors up to which two threads always win,
constexpr int kDfSplitSmall = 8;       // up to which on a lattice of at most,
constexpr int kDfSplitLarge = 12;      // up to which on one of more than
constexpr int kDfSplitSites = 12288;   // this many sites

bool df_split(int nv, int V) {
    return nv <= kDfSplit || (nv <= kDfSplitSmall ? V <= kDfSplitSites : nv <= kDfSplitLarge && V > kDfSplitSites);
}

template <int SPLIT>
__global__ void __launch_bounds__(kDfMaxThreads, 2) k_stencil_df(const dfc* __restrict__ U, Geom g, StencilDfSet s,
                                                              df kappa, df emu, df emu_inv) {
    extern __shared__ __align__(16) char smem[];
    const DfSmem S = df_carve(smem);
    const int site0 = blockIdx.x * kDfSites;
    const int site = min(site0 + (int)threadIdx.x, g.V - 1);
    pdl_trigger();
    df_stage(U, g, site0, S);   // (the links: nothing that a stream may still run here writes them)
    pdl_wait();
    const int v = threadIdx.y / SPLIT, half = threadIdx.y % SPLIT;
    if (v >= s.n_a + s.n_d) return;
    const int side = v < s.n_a ? 0 : 1;
    const int vi = side ? v - s.n_a : v;
    const dfc* in = (side ? s.in_d : s.in_a) + (size_t)vi * s.in_stride;
    // temporal weights: A uses (e^{mu}, e^{-mu}); A^dagger exchanges them
    const df wp_t = side ? emu_inv : emu, wm_t = side ? emu : emu_inv;
    DSpin acc;
#pragma unroll
    for (int a = 0; a < 3; ++a) acc.ur[a] = acc.ui[a] = acc.dr[a] = acc.di[a] = P2{0ull, 0ull};
#pragma unroll 1
    for (int pair = 0; pair < 2; ++pair) {   // x, y, then z, t
        const bool swap = pair == 0;
#pragma unroll 1
        for (int f = half; f < 2; f += SPLIT) df_hop<true>(acc, in, g.V, S, wp_t, wm_t, swap, f);
#pragma unroll 1
        for (int f = half; f < 2; f += SPLIT) df_hop<false>(acc, in, g.V, S, wp_t, wm_t, swap, f);
        if (swap) {   // the lower accumulators in their own lanes from here on
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                acc.dr[a] = p2_swp(acc.dr[a]);
                acc.di[a] = p2_swp(acc.di[a]);
            }
        }
    }
    if (SPLIT == 2) {   // this thread's spin pair (in ur, ui), summed over both senses
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const P2 gr = shfl_half(half ? acc.ur[a] : acc.dr[a]), gi = shfl_half(half ? acc.ui[a] : acc.di[a]);
            acc.ur[a] = p2_add(half ? acc.dr[a] : acc.ur[a], gr);
            acc.ui[a] = p2_add(half ? acc.di[a] : acc.ui[a], gi);
        }
    }
    if (site0 + (int)threadIdx.x >= g.V) return;
    const P2 K = {pk(kappa.hi, kappa.hi), pk(kappa.lo, kappa.lo)};
    P2 SR, SI;   // the scale 1/n_j (1/m_j), two-float from its FP64 value
    const bool scaled = s.scale != nullptr;
    if (scaled) {
        const double2 z = s.scale[(size_t)vi * kScalars + (side ? kScM : kScN)];
        const df zr = df_from_double(z.x), zi = df_from_double(z.y);
        SR = {pk(zr.hi, zr.hi), pk(zr.lo, zr.lo)};
        SI = {pk(zi.hi, zi.hi), pk(zi.lo, zi.lo)};
    }
    const float4* f = reinterpret_cast<const float4*>(in) + site;
    double2* out = (side ? s.out_d : s.out_a) + (size_t)vi * s.out_stride;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int q = 0; q < 2; q += SPLIT) {
            const int hf = SPLIT == 2 ? half : q;   // spins 2 hf, 2 hf + 1
            const int c0 = 6 * hf + a, c1 = c0 + 3;
            const float4 s0 = ld_after_wait(f + (size_t)c0 * g.V), s1 = ld_after_wait(f + (size_t)c1 * g.V);
            const P2 pr = {pk(s0.x, s1.x), pk(s0.y, s1.y)}, pi = {pk(s0.z, s1.z), pk(s0.w, s1.w)};
            const P2 kr = p2_prod(K, q ? acc.dr[a] : acc.ur[a]), ki = p2_prod(K, q ? acc.di[a] : acc.ui[a]);
            // gamma5 = diag(1, 1, -1, -1): upper spins psi - kappa acc, lower kappa acc - psi
            P2 orr = hf ? p2_add(kr, p2_neg(pr)) : p2_add(pr, p2_neg(kr));
            P2 oii = hf ? p2_add(ki, p2_neg(pi)) : p2_add(pi, p2_neg(ki));
            if (scaled) {   // (yr + i yi)(sr + i si)
                const P2 yr = orr, yi = oii;
                orr = p2_add(p2_prod(SR, yr), p2_prod(SI, p2_neg(yi)));
                oii = p2_add(p2_prod(SI, yr), p2_prod(SR, yi));
            }
            double r0, r1, i0, i1;
            p2_to_double(orr, r0, r1);
            p2_to_double(oii, i0, i1);
            out[s.out_abi ? (size_t)site * 12 + c0 : (size_t)c0 * g.V + site] = make_double2(r0, i0);
            out[s.out_abi ? (size_t)site * 12 + c1 : (size_t)c1 * g.V + site] = make_double2(r1, i1);
        }
    }
}

df df_of_host(double d) {
    df r;
    r.hi = (float)d;
    r.lo = (float)(d - (double)r.hi);
    return r;
}

}  // namespace

void stencil_df_init_attributes() {
    cudaFuncSetAttribute(k_stencil_df<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)df_smem());
    cudaFuncSetAttribute(k_stencil_df<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)df_smem());
}

void launch_stencil_df(const void* Udf, const Geom& g, const StencilDfSet& s, double kappa, double mu,
                       cudaStream_t st) {
    const int nv = s.n_a + s.n_d;
    if (nv == 0) return;
    const unsigned grid = (unsigned)((g.V + kDfSites - 1) / kDfSites);
#define NK_DF(SPLIT_)                                                                                        \
    launch_kernel(k_stencil_df<SPLIT_>, grid, dim3(kDfSites, SPLIT_ * nv), df_smem(), st, !s.scale, (const dfc*)Udf, \
                  g, s, df_of_host(kappa), df_of_host(exp(mu)), df_of_host(exp(-mu)))
    if (df_split(nv, g.V)) NK_DF(2);
    else NK_DF(1);
#undef NK_DF
}

}  // namespace nk

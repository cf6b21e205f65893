// Shared device helpers: complex arithmetic on float2/double2, deterministic
// block reductions, float <-> double conversions and two-float arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nk {

// ---- programmatic dependent launch ------------------------------------------------
// The operator entry points (stencils alone) are launched with `dependent`: a
// kernel's CTAs are placed, and stage the links, as soon as every CTA of the
// kernel before it in the stream has started and passed pdl_trigger; it touches
// no vector before pdl_wait, which returns once the kernels before it have
// completed and their writes are visible to ordinary loads.  It is alive while
// they still write, so its vectors are no read-only data of the grid: they are
// read by ordinary loads (no __ldg, no const __restrict__ pointer, which would
// also let the compiler move a load above the wait).  A caller that applies the operator again
// and again then has no launch gap and a filled last wave: FP32 stencil, 24 vectors at 10^4,
// 24.7 -> 21.9 us a call (one call alone, and the kernel inside a solve, take what they did).  Behind a kernel without pdl_trigger it is an ordinary launch.
// Inside an outer recurrence the kernels are launched plainly: there the
// waiting CTAs took slots unevenly (an outer step of 12 sources at 8^4 27.5 -> 30.7 us,
// 33 with an early trigger; 6^4, one source, 20.9 -> 22.6).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// An ordinary load that stays below a pdl_wait before it (volatile statements keep
// their order).
__device__ __forceinline__ float4 ld_after_wait(const float4* p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}
template <typename... P, typename... A>
inline void launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool dependent,
                          A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);   // an error is read by the caller's cudaGetLastError
}

template <typename R> struct C2;
template <> struct C2<float> { typedef float2 T; };
template <> struct C2<double> { typedef double2 T; };

__host__ __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__host__ __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }

__host__ __device__ __forceinline__ double2 cadd(double2 a, double2 b) { return mk(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 csub(double2 a, double2 b) { return mk(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * b as explicit fused multiply-adds: the same bits in every kernel (in a * b - c * d the
// compiler chooses which product it rounds)
__device__ __forceinline__ double2 cmul_fma(double2 a, double2 b) {
    return mk(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__host__ __device__ __forceinline__ double2 cconj(double2 a) { return mk(a.x, -a.y); }
__host__ __device__ __forceinline__ double2 cscale(double2 a, double s) { return mk(a.x * s, a.y * s); }
__host__ __device__ __forceinline__ double cabs1(double2 a) { return fabs(a.x) + fabs(a.y); }
__host__ __device__ __forceinline__ double cnorm2(double2 a) { return a.x * a.x + a.y * a.y; }
__host__ __device__ __forceinline__ double2 cinv(double2 a) {
    // 1/a with Smith's scaling to avoid overflow in |a|^2
    if (fabs(a.x) >= fabs(a.y)) {
        double r = a.y / a.x, d = a.x + a.y * r;
        return mk(1.0 / d, -r / d);
    } else {
        double r = a.x / a.y, d = a.x * r + a.y;
        return mk(r / d, -1.0 / d);
    }
}
__host__ __device__ __forceinline__ double2 cdiv(double2 a, double2 b) { return cmul(a, cinv(b)); }
// sqrt(x) and 1 / sqrt(x) of a positive finite x from one reciprocal square
// root (410 clocks; a square root takes 650, a division 620): y = rsqrt(x),
// then one Newton correction of x y.
__device__ __forceinline__ double sqrt_inv(double x, double& inv) {
    const double y = rsqrt(x), s = x * y;
    inv = y;
    return fma(0.5 * y, fma(-s, s, x), s);
}

// beta = sqrt(delta) (principal branch), gamma = delta^* / beta, 1 / beta and
// 1 / gamma of a finite delta != 0, without a division: with d = delta / 2^e
// (e even, exact, so that max(|Re d|, |Im d|) is in [1, 4)), m = |d| and
// 1 / m come from one reciprocal square root, the parts of sqrt(d) from a
// second; then 1 / beta = beta^* / |delta|, gamma = (delta beta)^* / |delta| and
// 1 / gamma = delta beta / |delta|^2.
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }   // |e| <= 1022
__device__ __forceinline__ void csqrt_scalars(double2 delta, double2& beta, double2& gamma, double2& inv_beta,
                                              double2& inv_gamma) {
    const int hx = __double2hiint(delta.x) & 0x7fffffff, hy = __double2hiint(delta.y) & 0x7fffffff;
    const int e = min(max(((max(hx, hy) >> 20) - 1023) & ~1, -1022), 1022);
    const double sc = pow2(-e), up = pow2(e >> 1), down = pow2(-(e >> 1));
    const double2 d = mk(delta.x * sc, delta.y * sc);
    double im;
    const double m = sqrt_inv(fma(d.x, d.x, d.y * d.y), im);
    double iv;
    const double t = sqrt_inv(0.5 * (m + fabs(d.x)), iv), o = 0.5 * d.y * iv;
    // (t, o) for Re d >= 0, else (|o|, sign(Im d) t)
    const double2 b = d.x >= 0.0 ? mk(t, o) : mk(fabs(o), d.y >= 0.0 ? t : -t);
    const double2 w = cscale(cmul_fma(d, b), im);
    beta = cscale(b, up);
    gamma = cscale(cconj(w), up);
    inv_beta = cscale(cconj(b), im * down);
    inv_gamma = cscale(w, im * down);
}

__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) { return mk(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return mk(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Warp sum of a double2 in a fixed butterfly order (deterministic).
__device__ __forceinline__ double2 warp_sum(double2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Linear thread index and thread count of the block (blocks may be 2-D with
// blockDim.x a multiple of 32: warps are then runs of 32 linear indices).
__device__ __forceinline__ int block_tid() { return threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z); }
__device__ __forceinline__ int block_threads() { return blockDim.x * blockDim.y * blockDim.z; }

// Warp sum of a double2 for a reduction tail: in the first exchange the lower
// half-warp keeps the real parts and the upper half the imaginary ones, so
// each level costs one FP64 addition instead of two (an FP64 warp instruction
// holds its pipe 64 clocks on GB300 whatever its active lanes).  x in lanes
// 0-15, y in lanes 16-31.
__device__ __forceinline__ double warp_sum_split(double2 v) {
    const bool up = (block_tid() & 16) != 0;
    const double got = __shfl_xor_sync(0xffffffffu, up ? v.x : v.y, 16);
    double t = (up ? v.y : v.x) + got;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Block sum of a double2 (<= 1024 threads in whole warps). Every thread of the
// block receives the same value; the summation order is fixed.  Only warp 0
// does the second level (FP64 adds are scarce on GB300), real parts in the
// lower half-warp and imaginary ones in the upper; the result is broadcast
// through shared memory.  The butterfly of the second level stops at the
// number of warps (lanes beyond it hold zeros).
__device__ __forceinline__ double2 block_sum(double2 v, double2* sh /* >= 33 */) {
    const double s = warp_sum_split(v);
    const int tid = block_tid();
    int lane = tid & 31, w = tid >> 5, nw = block_threads() >> 5;
    double* f = reinterpret_cast<double*>(sh);
    const int q = lane & 15, part = lane >> 4;   // warp q (and q + 16), real or imaginary part
    __syncthreads();
    if (q == 0) f[2 * w + part] = s;
    __syncthreads();
    if (w == 0) {
        double t = q < nw ? f[2 * q + part] : 0.0;
        if (nw > 16 && q + 16 < nw) t += f[32 + 2 * q + part];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
            if (o < nw) t += __shfl_xor_sync(0xffffffffu, t, o);   // only the levels that combine real partials
        if (q == 0) f[64 + part] = t;
    }
    __syncthreads();
    return sh[32];
}
__device__ __forceinline__ double block_sum(double v, double* sh /* >= 32 */) {
    v = warp_sum(v);
    const int tid = block_tid();
    int lane = tid & 31, w = tid >> 5, nw = block_threads() >> 5;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = lane < nw ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (o < nw) t += __shfl_xor_sync(0xffffffffu, t, o);
    // lanes below the next power of two of nw hold the sum
    return __shfl_sync(0xffffffffu, t, 0);
}

// Two-stage deterministic reduction, stage 1: thread 0 of each block writes
// its block's partial; the block that arrives last (integer ticket, no
// floating-point atomics) returns true and finishes the sum in fixed order.
__device__ __forceinline__ bool finish_partial(double2 part, double2* partials, unsigned* counter,
                                               int slot, int nslots) {
    __shared__ bool last;
    if (block_tid() == 0) {
        partials[slot] = part;
        __threadfence();
        unsigned ticket = atomicAdd(counter, 1u);
        last = (ticket == (unsigned)nslots - 1u);
    }
    __syncthreads();
    return last;
}

// Stage 2: fixed-order sum of the nslots partials (all threads of the last
// block).  Four loads in flight per thread: the tail of a step waits for them.
__device__ __forceinline__ double2 sum_partials(const double2* partials, int nslots, double2* sh) {
    __threadfence();
    double2 a = mk(0.0, 0.0);
    const int T = block_threads();
    for (int i0 = block_tid(); i0 < nslots; i0 += 4 * T) {
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = i0 + u * T < nslots ? __ldcg(partials + i0 + u * T) : mk(0.0, 0.0);
        if (i0 + T < nslots) {
            v[0] = cadd(v[0], v[1]);
            if (i0 + 2 * T < nslots) v[0] = cadd(v[0], cadd(v[2], v[3]));
        }
        a = i0 < T ? v[0] : cadd(a, v[0]);
    }
    return block_sum(a, sh);
}

// ---- float <-> double on the integer pipe ---------------------------------------
// On GB300 the FP64 pipe is 1/64 of the FP32 rate and cvt.f64.f32 /
// cvt.f32.f64 issue on it too, so the hot kernels move between the formats
// with integer bit operations only (IEEE 754 binary32 <-> binary64 field
// layout), with no conversion instruction even on a predicated-off path.
// Normal numbers and zero convert exactly / round to nearest; the edge cases
// the vectors of this method never reach are mapped without a conversion
// instruction: float subnormals and double results below the normal float
// range become signed zero, overflow becomes infinity, NaN stays NaN.

// float -> double, exact for normal floats and zero
__device__ __forceinline__ double f2d_int(float f) {
    const unsigned u = __float_as_uint(f);
    const unsigned s = u & 0x80000000u;
    const unsigned a = u & 0x7fffffffu;
    unsigned hi = s | ((a >> 3) + (896u << 20));
    unsigned lo = a << 29;
    if (a < 0x00800000u) { hi = s; lo = 0u; }                        // zero, subnormal -> 0
    if (a >= 0x7f800000u) { hi = s | 0x7ff00000u | ((a >> 3) & 0x000fffffu); }   // inf / NaN
    return __hiloint2double((int)hi, (int)lo);
}

// double -> float, rounded to nearest (ties away from zero in magnitude; ties
// occur with probability 2^-29 and differ from round-to-even by one ulp).
// Every range check is made on the 32-bit high word: checks on the 64-bit
// pattern of |d| were turned by the compiler into FP64 comparisons, which
// issue on the scarce FP64 pipe.
__device__ __forceinline__ float d2f_int(double d) {
    const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
    const unsigned s = h & 0x80000000u, ah = h & 0x7fffffffu;
    // (wraps around below the normal float range; the underflow rule is applied last)
    const unsigned t = (((ah - (896u << 20)) << 3) | (l >> 29)) + ((l >> 28) & 1u);
    unsigned r = t;
    if (ah >= (1151u << 20) || t >= (255u << 23)) r = 0x7f800000u;             // overflow -> inf
    if (ah < (897u << 20)) r = 0u;                                               // below normal floats -> 0
    if (ah > 0x7ff00000u || (ah == 0x7ff00000u && l != 0u)) r = 0x7fc00000u;     // NaN
    return __uint_as_float(s | r);
}

// double -> (hi, lo) floats with hi + lo == d to about 2^-48 relative: hi is d
// truncated to 24 significant bits (exact in float), lo the remaining 29 bits
// rounded to a float.  Outside the normal float range: (d2f_int(d), 0).
__device__ __forceinline__ float2 d2ff_int(double d) {
    const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
    const unsigned s = h & 0x80000000u, ah = h & 0x7fffffffu;
    const unsigned e = ah >> 20;
    const bool normal = ah >= (897u << 20) && ah < (1151u << 20);
    float hi = __uint_as_float(s | (((ah - (896u << 20)) << 3) | (l >> 29)));
    const unsigned mlo = l & 0x1fffffffu;                                        // d - hi = mlo * 2^(e - 1075)
    float lo = __uint2float_rn(mlo) * __uint_as_float(((e > 948u ? e : 949u) - 948u) << 23);
    lo = __uint_as_float(__float_as_uint(lo) | s);
    if (e <= 948u) lo = 0.0f;
    if (!normal) { hi = d2f_int(d); lo = 0.0f; }
    return make_float2(hi, lo);
}

// ---- two-float ("df") arithmetic ---------------------------------------------------
// A value is hi + lo with |lo| <= ulp(hi); about 48 significant bits, computed
// on the FP32 pipe with the error-free transformations TwoSum (Knuth) and
// TwoProd via FMA (the double-float arithmetic of Dekker and of Hida, Li and
// Bailey's double-double library).  The _rn intrinsics keep the compiler from
// contracting or reassociating the steps.
struct df {
    float hi, lo;
    __host__ __device__ __forceinline__ df() {}
    __host__ __device__ __forceinline__ df(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ __forceinline__ df(int v) : hi((float)v), lo(0.0f) {}
};
__device__ __forceinline__ df df_fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return df(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ df operator+(df a, df b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float v = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    return df_fast_two_sum(s, e);
}
__device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}
__device__ __forceinline__ df& operator+=(df& a, df b) { a = a + b; return a; }
__device__ __forceinline__ df df_from_double(double d) {
    const float2 p = d2ff_int(d);
    return df(p.x, p.y);
}
__device__ __forceinline__ double df_to_double(df a) { return f2d_int(a.hi) + f2d_int(a.lo); }

struct __align__(16) dfc {
    df x, y;
};

// Unnormalised two-float accumulator: the value is s + e, with |e| small
// against |s| but not renormalised after each step.  Adding an exact product
// (TwoProd via FMA, including the cross terms of two-float operands) or
// another value is TwoSum on the leading parts and a plain FP32 sum of the
// trailing parts: 12 and 8 FP32 instructions, against 18 and 11 for the
// normalised product and sum (the accumulation of Ogita, Rump and Oishi's
// compensated dot product, applied to two-float operands).  dfa_value
// renormalises once at the end.
struct dfa {
    float s, e;
};
__device__ __forceinline__ dfa dfa_of(df a) { return {a.hi, a.lo}; }
__device__ __forceinline__ dfa dfa_neg(dfa a) { return {-a.s, -a.e}; }
// (ah + al) (bh + bl) up to the al bl term
__device__ __forceinline__ dfa dfa_prod(float ah, float al, float bh, float bl) {
    const float p = __fmul_rn(ah, bh);
    float e = __fmaf_rn(ah, bh, -p);
    e = __fmaf_rn(ah, bl, e);
    e = __fmaf_rn(al, bh, e);
    return {p, e};
}
// a += s + e
__device__ __forceinline__ void dfa_add(dfa& a, float s, float e) {
    const float t = __fadd_rn(a.s, s);
    const float v = __fsub_rn(t, a.s);
    const float err = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, v)), __fsub_rn(s, v));
    a.s = t;
    a.e = __fadd_rn(a.e, __fadd_rn(e, err));
}
__device__ __forceinline__ void dfa_add(dfa& a, dfa b) { dfa_add(a, b.s, b.e); }
__device__ __forceinline__ void dfa_add_prod(dfa& a, float ah, float al, float bh, float bl) {
    const dfa p = dfa_prod(ah, al, bh, bl);
    dfa_add(a, p.s, p.e);
}
__device__ __forceinline__ df dfa_value(dfa a) { return df_fast_two_sum(a.s, a.e); }
struct dfac {
    dfa x, y;
};
template <> struct C2<df> { typedef dfc T; };
static_assert(sizeof(dfc) == 16, "two-float complex is 16 bytes");

}  // namespace nk

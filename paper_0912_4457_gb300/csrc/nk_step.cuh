// The scalars between two outer steps, shared by the kernels that finish a step
// (lanczos.cu, stencil64.cu).
#pragma once

#include "nk_common.cuh"
#include "nk_kernels.h"

namespace nk {

template <bool TS>
__device__ __forceinline__ StepScalars step_scalars(double2 d) {
    StepScalars t;
    t.inv_beta = t.inv_gamma = mk(0.0, 0.0);
    if (!TS) {
        // beta <- sqrt(r^dag r)
        t.ok = d.x > 0.0 && isfinite(d.x);
        double inv = 0.0;
        const double b = t.ok ? sqrt_inv(d.x, inv) : sqrt(d.x);
        t.beta = t.gamma = mk(b, 0.0);
        t.inv_beta = t.inv_gamma = mk(inv, 0.0);
    } else if ((d.x == 0.0 && d.y == 0.0) || !isfinite(d.x) || !isfinite(d.y)) {
        // serious breakdown: delta = 0 (App. B); a non-finite delta is treated alike
        t.beta = t.gamma = mk(0.0, 0.0);
        t.ok = false;
    } else {
        // beta <- sqrt(delta), gamma <- delta^* / beta
        csqrt_scalars(d, t.beta, t.gamma, t.inv_beta, t.inv_gamma);
        t.ok = true;
    }
    return t;
}

// Scalars of step j + 1 from those of step j (1/n_j, 1/m_j): n_{j+1} = beta_j,
// m_{j+1} = gamma_j^*.
template <bool TS>
__device__ __forceinline__ void next_scalars(double2* sc, const StepScalars& t) {
    const double2 inv_n = sc[kScN], inv_m = sc[kScM];
    sc[kScN] = t.inv_beta;
    sc[kScC1] = cmul_fma(t.gamma, inv_n);           // gamma (Hermitian: beta) / n_j
    sc[kScD] = t.inv_gamma;
    sc[kScM] = cconj(t.inv_gamma);
    sc[kScC1L] = cmul_fma(cconj(t.beta), inv_m);
}

}  // namespace nk

// Roberts-Higham iteration of the nested method, per RHS (App. C step 5, Eq.
// Roberts): S <- (S + S^{-1})/2 on the dense H_l until it stops moving, and
// c = V_l sgn(H_l) e_1.  (Steps 3-4, the LU and the inner Lanczos, are in
// inner_lanczos.cu.)  In the Hermitian case (mu = 0) it is real arithmetic.
//
// RHi runs one thread-block cluster per RHS: the rows of the l x l matrix
// being inverted (in-place Gauss-Jordan with partial pivoting and row
// interchanges) are spread cyclically over the cluster's CTAs and held in
// their shared memory; the pivot search, the pivot row broadcast and the row
// interchange go through distributed shared memory, with one cluster barrier
// per pivot (candidate rows published in buffers that alternate between
// pivots).
#include <cooperative_groups.h>

#include "inner_arith.cuh"
#include "nk_kernels.h"

namespace cg = cooperative_groups;

namespace nk {

namespace {

// ---- Roberts-Higham iteration on H_l, one cluster per RHS ----------------------

constexpr int kRhiThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kRhiThreads) k_rhi(Inner in, int C, int maxit, double stop) {
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int rhs = blockIdx.x / C;
    const int L = in.ell;
    const int nloc = (L - rank + C - 1) / C;       // rows rank, rank + C, ...
    const int nmax = (L + C - 1) / C;
    extern __shared__ __align__(16) unsigned char smem[];
    T* M = reinterpret_cast<T*>(smem);              // [nmax][L]
    T* prow = M + (size_t)nmax * L;                 // [L]
    T* tmp = prow + L;                              // [L]
    T* cand_row = tmp + L;                          // [2][L] published candidate pivot row
    T* rowc = cand_row + 2 * L;                     // [2][L] published row c
    T* fcol = rowc + 2 * L;                         // [nmax]
    int* piv = reinterpret_cast<int*>(fcol + nmax); // [L]
    __shared__ double cand_val[2];
    __shared__ int cand_idx[2];
    __shared__ double part[2];
    __shared__ double sh1[32];
    __shared__ int s_stop;

    const int status0 = in.status[rhs];   // identical in every CTA of the cluster
    T* S = reinterpret_cast<T*>(in.S) + (size_t)rhs * L * L;
    const double2* alo = in.al + (size_t)rhs * L;
    const double2* blo = in.bl + (size_t)rhs * L;
    const double2* glo = in.gl + (size_t)rhs * L;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;

    // S_0 = H_l (own rows)
    for (int e = tid; e < nloc * L; e += blockDim.x) {
        int li = e / L, col = e % L, i = rank + C * li;
        T v = t_zero(T());
        if (status0 == kStatusOK) {
            if (col == i) v = t_from(alo[i], T());
            else if (col == i - 1) v = t_from(blo[i - 1], T());
            else if (col == i + 1) v = t_from(glo[i], T());
        }
        S[(size_t)i * L + col] = v;
    }
    int iters = 0;
    bool ok = status0 == kStatusOK;
    bool converged = false;
    for (int it = 1; ok && it <= maxit; ++it) {
        iters = it;
        for (int e = tid; e < nloc * L; e += blockDim.x) {
            int li = e / L, col = e % L;
            M[(size_t)li * L + col] = S[(size_t)(rank + C * li) * L + col];
        }
        __syncthreads();
        // ---- in-place Gauss-Jordan inverse of M with partial pivoting ----
        // One cluster barrier per pivot: each CTA publishes its candidate pivot
        // row (and the owner of row c that row) in a buffer of parity c & 1
        // before the barrier; after it every CTA reads the pivot row and row c
        // from those buffers, which their owners rewrite only two pivots later,
        // after every CTA has passed the next barrier.
        for (int c = 0; c < L; ++c) {
            const int par = c & 1;
            // (a) local candidate: largest |M(i,c)|^2 over own rows i >= c (lowest i on ties);
            // nloc <= 32, so warp 0 holds one row per lane
            if (warp == 0) {
                double bv = -1.0;
                int bi = 0x7fffffff;
                if (lane < nloc) {
                    const int i = rank + C * lane;
                    if (i >= c) { bv = t_norm2(M[(size_t)lane * L + c]); bi = i; }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    double ov = __shfl_xor_sync(0xffffffffu, bv, o);
                    int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
                }
                if (lane == 0) { cand_val[par] = bv; cand_idx[par] = bi; }
            }
            __syncthreads();
            if (cand_val[par] >= 0.0) {
                const T* src = M + (size_t)((cand_idx[par] - rank) / C) * L;
                for (int col = tid; col < L; col += blockDim.x) cand_row[par * L + col] = src[col];
            }
            if (c % C == rank) {
                const T* src = M + (size_t)(c / C) * L;
                for (int col = tid; col < L; col += blockDim.x) rowc[par * L + col] = src[col];
            }
            cl.sync();                                                  // the one barrier of the pivot
            // (b) pivot row over the cluster, ranks in fixed order (same decision everywhere)
            double pv = -1.0;
            int pi = 0x7fffffff;
            for (int q = 0; q < C; ++q) {
                double qv = cl.map_shared_rank(cand_val, q)[par];
                int qi = cl.map_shared_rank(cand_idx, q)[par];
                if (qv > pv || (qv == pv && qi < pi)) { pv = qv; pi = qi; }
            }
            if (!(pv > 0.0)) {              // singular (same decision in every CTA)
                ok = false;
                cl.sync();                  // no CTA leaves while others read its buffers
                break;
            }
            if (tid == 0) piv[c] = pi;
            // (c) fetch the pivot row and, for the owner of row pi, old row c
            {
                const T* src = cl.map_shared_rank(cand_row, pi % C) + par * L;
                for (int col = tid; col < L; col += blockDim.x) prow[col] = src[col];
                if (pi != c && pi % C == rank) {
                    const T* srcc = cl.map_shared_rank(rowc, c % C) + par * L;
                    for (int col = tid; col < L; col += blockDim.x) tmp[col] = srcc[col];
                }
            }
            __syncthreads();
            const T pinv = t_inv(prow[c]);
            // (d) multipliers of the own rows other than the pivot row, already
            // divided by the pivot (the row in slot pi now holds old row c)
            for (int li = tid; li < nloc; li += blockDim.x) {
                const int i = rank + C * li;
                const T f = (i == pi && pi != c) ? tmp[c] : M[(size_t)li * L + c];
                fcol[li] = i == c ? t_zero(T()) : t_mul(f, pinv);
            }
            __syncthreads();
            // (e) rows by warp, columns by lane: the pivot row scaled into slot c;
            // every other row: M(i,:) -= f' prow, M(i,c) = -f'
            for (int li = warp; li < nloc; li += nwarps) {
                const int i = rank + C * li;
                T* row = M + (size_t)li * L;
                if (i == c) {
                    for (int col = lane; col < L; col += 32) row[col] = col == c ? pinv : t_mul(prow[col], pinv);
                } else {
                    const T* src = (i == pi && pi != c) ? tmp : row;
                    const T f = fcol[li];
                    for (int col = lane; col < L; col += 32)
                        row[col] = col == c ? t_neg(f) : t_fma(t_neg(f), prow[col], src[col]);
                }
            }
            __syncthreads();
        }
        if (!ok) break;
        // undo the interchanges on the columns of the inverse
        for (int c = L - 1; c >= 0; --c) {
            int q = piv[c];
            if (q != c) {
                for (int li = tid; li < nloc; li += blockDim.x) {
                    T a = M[(size_t)li * L + c];
                    M[(size_t)li * L + c] = M[(size_t)li * L + q];
                    M[(size_t)li * L + q] = a;
                }
            }
            __syncthreads();
        }
        // S <- (S + S^{-1}) / 2 and the relative Frobenius change
        double dsum = 0.0, nsum = 0.0;
        for (int e = tid; e < nloc * L; e += blockDim.x) {
            int li = e / L, col = e % L;
            size_t gi = (size_t)(rank + C * li) * L + col;
            T so = S[gi];
            T sn = t_scale(t_add(so, M[(size_t)li * L + col]), 0.5);
            dsum += t_norm2(t_sub(sn, so));
            nsum += t_norm2(sn);
            S[gi] = sn;
        }
        dsum = block_sum(dsum, sh1);
        nsum = block_sum(nsum, sh1);
        if (tid == 0) { part[0] = dsum; part[1] = nsum; }
        cl.sync();
        double dt = 0.0, nt = 0.0;
        for (int q = 0; q < C; ++q) {
            const double* pq = cl.map_shared_rank(part, q);
            dt += pq[0];
            nt += pq[1];
        }
        cl.sync();   // every CTA has read the partials before they are rewritten
        if (sqrt(dt) <= stop * sqrt(nt)) { converged = true; break; }
    }
    if (tid == 0) s_stop = 0;
    __syncthreads();
    // s = S e_1 (own rows), iteration count, status
    for (int li = tid; li < nloc; li += blockDim.x) {
        int i = rank + C * li;
        in.s[(size_t)rhs * L + i] = t_to2(S[(size_t)i * L]);
    }
    if (rank == 0 && tid == 0) {
        in.rhi_iters[rhs] = iters;
        if (status0 == kStatusOK && !converged) in.status[rhs] = kStatusRhi;
    }
}

// c = V_l s (k-vector per RHS)
__global__ void k_combine(Inner in) {
    const int rhs = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= in.k) return;
    double2* c = in.c + (size_t)rhs * (in.kstride > 0 ? in.kstride : in.k);
    if (in.status[rhs] != kStatusOK) { c[i] = mk(0.0, 0.0); return; }
    const double2* Vl = in.Vl + (size_t)rhs * in.ell * in.k;
    const double2* s = in.s + (size_t)rhs * in.ell;
    double2 acc = mk(0.0, 0.0);
    for (int j = 0; j < in.ell; ++j) acc = cadd(acc, cmul(Vl[(size_t)j * in.k + i], s[j]));
    c[i] = acc;
}

}  // namespace

// Largest dynamic shared memory any RHi launch needs (l <= 256, complex, 8 CTAs).
static size_t rhi_smem_max();

void init_kernel_attributes() {
    inner_lanczos_init_attributes();
    cudaFuncSetAttribute(k_rhi<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rhi_smem_max());
    cudaFuncSetAttribute(k_rhi<double2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rhi_smem_max());
    cudaFuncSetAttribute(k_rhi<double>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaFuncSetAttribute(k_rhi<double2>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    stencil32_init_attributes();
    stencil_df_init_attributes();
}

static int rhi_cluster_size(int ell) { return ell >= 64 ? 8 : (ell >= 16 ? 4 : 1); }

template <typename T>
static size_t rhi_smem(int ell, int C) {
    int nmax = (ell + C - 1) / C;
    return (size_t)nmax * ell * sizeof(T) + 6 * (size_t)ell * sizeof(T) + (size_t)nmax * sizeof(T) +
           (size_t)ell * sizeof(int) + 16;
}

static size_t rhi_smem_max() { return rhi_smem<double2>(256, 8); }

template <typename T>
static cudaError_t launch_rhi_t(const Inner& in, cudaStream_t st) {
    const int C = rhi_cluster_size(in.ell);
    size_t smem = rhi_smem<T>(in.ell, C);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(in.n_rhs * C);
    cfg.blockDim = dim3(kRhiThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_rhi<T>, in, C, 50, 1e-10);
}

int launch_rhi(const Inner& in, cudaStream_t st) {
    // RHi stays FP64 in every schedule: near the imaginary axis sgn is ill
    // conditioned and the iteration amplifies the working precision's rounding
    // (two-float RHi left 2 of 12 sources of the 16^3 x 32 test at 2.5e-8)
    return (int)(in.two_sided ? launch_rhi_t<double2>(in, st) : launch_rhi_t<double>(in, st));
}

void launch_inner_combine(const Inner& in, cudaStream_t st) {
    dim3 grid((in.k + 127) / 128, in.n_rhs);
    k_combine<<<grid, 128, 0, st>>>(in);
}

}  // namespace nk

// Roberts-Higham iteration of the nested method, per RHS (App. C step 5, Eq.
// Roberts): S <- (S + S^{-1})/2 on the dense H_l until it stops moving, and
// c = V_l sgn(H_l) e_1.  (Steps 3-4, the LU and the inner Lanczos, are in
// inner_lanczos.cu.)  In the Hermitian case (mu = 0) it is real arithmetic.
//
// RHi runs one thread-block cluster per RHS: the rows of the l x l matrix
// being inverted (in-place Gauss-Jordan with partial pivoting and row
// interchanges) are spread cyclically over the cluster's CTAs and held in
// their shared memory.
//
// What bounds it: a pivot is a rank-1 update of the whole matrix (l^2 / C
// complex multiply-adds per CTA: 4096 clocks of the FP64 pipe at l = 128, C = 8)
// and a chain of dependent steps -- multipliers, the next column, the pivot
// search, the inverse of the pivot, the exchange through the cluster.  Run one after the other
// (the earlier form: 8 us per pivot at l = 128) the chain costs as much again
// as the update, so here it runs one pivot ahead: four warps per CTA form the
// next pivot column from the rows as they are, choose their candidate, update
// and publish its row (and row c + 1) and arrive at the cluster barrier; then
// they wait for it and fetch the pivot row, while seven warps are still
// updating the other rows for the present pivot.  Measured: 12 two-sided RHS,
// l = 128 6.2 -> 3.5 ms; the inner part of 12 Hermitian ones at k = 768, l = 160 8.2 ->
// 5.2 ms, of one at l = 64, k = 256 2.8 -> 1.8 (both with the cluster Lanczos).
#include <cooperative_groups.h>

#include "inner_arith.cuh"
#include "nk_kernels.h"

namespace cg = cooperative_groups;

namespace nk {

namespace {

// ---- Roberts-Higham iteration on H_l, one cluster per RHS ----------------------

// Warps 0-3: the pivot chain (0: multipliers, next column, search, inverse of the
// candidate; 1-3: the published rows); warps 4-7 and 9-11: the update.  An SM
// sub-partition (warp index mod 4) has one FP64 pipe: warp 8 stays idle so that
// warp 0 shares its pipe with one updating warp instead of two.
constexpr int kRhiChain = 4, kRhiBulk = 7;
constexpr int kRhiThreads = 32 * 12;
constexpr int kRhiEarly = 2;     // items per updating warp before the next pivot is known
constexpr int kRhiMaxC = 16;

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// |x|^2 as an ordered key: 0 unless it is positive (zero and NaN are no pivot)
template <typename T>
__device__ __forceinline__ unsigned long long pivot_key(T x) {
    const unsigned long long b = abs_bits(t_norm2(x));
    return b <= 0x7ff0000000000000ull ? b : 0ull;
}

template <typename T>
__global__ void __launch_bounds__(kRhiThreads) k_rhi(Inner in, int C, int maxit, double stop) {
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int rhs = blockIdx.x / C;
    const int L = in.ell, LD = L + 1;               // padded rows: a column of the CTA's rows is conflict-free
    const int nloc = (L - rank + C - 1) / C;       // rows rank, rank + C, ... (at most 32)
    const int nmax = (L + C - 1) / C;
    extern __shared__ __align__(16) unsigned char smem[];
    T* M = reinterpret_cast<T*>(smem);              // [nmax][LD]
    T* prow = M + (size_t)nmax * LD;                // [2][L] pivot row of the present and the next pivot
    T* cand_row = prow + 2 * L;                     // [2][L] published candidate pivot row
    T* rowc = cand_row + 2 * L;                     // [2][L] published row c
    T* fcol = rowc + 2 * L;                         // [nmax]
    __shared__ unsigned long long cand_key[2][kRhiMaxC];
    __shared__ int cand_idx[2][kRhiMaxC];
    __shared__ T cand_inv[2][kRhiMaxC];
    __shared__ double part[2][kRhiMaxC][2];
    __shared__ double sh1[32];
    __shared__ int s_li;                            // own candidate (local row) of the next pivot, or -1
    __shared__ int s_pi;                            // present pivot row (-1: singular)

    const int status0 = in.status[rhs];   // identical in every CTA of the cluster
    T* S = reinterpret_cast<T*>(in.S) + (size_t)rhs * L * L;
    const double2* alo = in.al + (size_t)rhs * L;
    const double2* blo = in.bl + (size_t)rhs * L;
    const double2* glo = in.gl + (size_t)rhs * L;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const bool chain = warp < kRhiChain;
    const int nb = (L + 31) / 32;                   // column blocks

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
    // warp 0: this CTA's candidate for pivot row c, x = M(i, c) of own row `lane`
    // (i >= c, else no candidate): largest |x|^2, lowest row on ties
    // (all lanes return its value and key)
    auto search = [&](int c, T x, unsigned long long& key) -> T {
        const int i = rank + C * lane;
        key = lane < nloc && i >= c ? pivot_key(x) : 0ull;
        int bi = lane < nloc && i >= c ? lane : 0x7fffffff;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(kFull, key, o);
            const int oi = __shfl_xor_sync(kFull, bi, o);
            if (ok > key || (ok == key && oi < bi)) { key = ok; bi = oi; }
        }
        const bool any = bi != 0x7fffffff;
        if (lane == 0) s_li = any ? bi : -1;
        return shfl_from(x, any ? bi : 0);
    };
    // warp 0: the candidate (value x, local row li or -1) to every CTA
    auto publish = [&](int par, T x, unsigned long long key, int li) {
        const T inv = key ? pivot_inv(x) : t_zero(T());
        if (lane < C) {
            *cl.map_shared_rank(&cand_key[par][rank], lane) = key;
            *cl.map_shared_rank(&cand_idx[par][rank], lane) = li >= 0 ? rank + C * li : 0x7fffffff;
            *cl.map_shared_rank(&cand_inv[par][rank], lane) = inv;
        }
    };
    int iters = 0;
    bool ok = status0 == kStatusOK;
    bool converged = false;
    for (int it = 1; ok && it <= maxit; ++it) {
        iters = it;
        __syncthreads();
        for (int e = tid; e < nloc * L; e += blockDim.x) {
            int li = e / L, col = e % L;
            M[(size_t)li * LD + col] = S[(size_t)(rank + C * li) * L + col];
        }
        int perm = tid;   // thread j < l: column of the interchanged inverse that holds column j
        __syncthreads();
        // ---- in-place Gauss-Jordan inverse of M with partial pivoting ----
        // pivot 0: candidates from the matrix as it is
        if (warp == 0) {
            unsigned long long key;
            const T x = search(0, lane < nloc ? M[(size_t)lane * LD] : t_zero(T()), key);
            __syncwarp();
            publish(0, x, key, s_li);
        }
        __syncthreads();
        for (int col = tid; col < L; col += blockDim.x) {
            if (s_li >= 0) cand_row[col] = M[(size_t)s_li * LD + col];
            if (rank == 0) rowc[col] = M[col];
        }
        cluster_arrive();
        for (int c = 0; c < L; ++c) {
            const int par = c & 1;
            T* pr = prow + par * L;
            cluster_wait();
            int pi = -1;
            if (chain) {
                // the pivot row over the cluster (same decision everywhere), fetched;
                // the slot of row pi takes old row c
                unsigned long long key = lane < C ? cand_key[par][lane] : 0ull;
                int bi = lane < C ? cand_idx[par][lane] : 0x7fffffff;
#pragma unroll
                for (int o = kRhiMaxC / 2; o > 0; o >>= 1) {
                    if (o >= C) continue;
                    const unsigned long long ok2 = __shfl_xor_sync(kFull, key, o);
                    const int oi = __shfl_xor_sync(kFull, bi, o);
                    if (ok2 > key || (ok2 == key && oi < bi)) { key = ok2; bi = oi; }
                }
                key = __shfl_sync(kFull, key, 0);
                pi = key ? __shfl_sync(kFull, bi, 0) : -1;
                if (tid == 0) s_pi = pi;
                if (pi >= 0) {
                    const T* src = cl.map_shared_rank(cand_row, pi % C) + par * L;
                    for (int col = tid; col < L; col += 32 * kRhiChain) pr[col] = src[col];
                    if (pi != c && pi % C == rank) {
                        const T* srcc = cl.map_shared_rank(rowc, c % C) + par * L;
                        T* row = M + (size_t)((pi - rank) / C) * LD;
                        for (int col = tid; col < L; col += 32 * kRhiChain) row[col] = srcc[col];
                    }
                }
            }
            __syncthreads();   // pivot row in place; the update for pivot c - 1 is complete
            pi = s_pi;
            if (pi < 0) { ok = false; break; }     // singular (same decision in every CTA)
            if (perm == c) perm = pi;
            else if (perm == pi) perm = c;
            const T pinv = cand_inv[par][pi % C];
            // multipliers of the own rows, already divided by the pivot
            T f = t_zero(T());
            if (warp == 0) {
                const int i = rank + C * lane;
                if (lane < nloc && i != c) f = t_mul(M[(size_t)lane * LD + c], pinv);
                if (lane < nloc) fcol[lane] = f;
            }
            __syncthreads();
            const bool own_c = c % C == rank;
            const int done = c > rank ? (c - rank + C - 1) / C : 0;   // own rows i < c
            const bool own_n = (c + 1) % C == rank && c + 1 < L;
            const int ln = own_n ? (c + 1 - rank) / C : -1;           // local row of row c + 1
            // row li, column block cb: M(i,:) -= f prow, M(i,c) = -f
            auto update = [&](int li, int cb, bool out) {
                const int col = cb * 32 + lane;
                if (col >= L) return;
                T* m = M + (size_t)li * LD + col;
                const T nf = t_neg(fcol[li]);
                const T v = col == c ? nf : t_fma(nf, pr[col], *m);
                *m = v;
                if (out) {
                    if (li == s_li) cand_row[(par ^ 1) * L + col] = v;
                    if (li == ln) rowc[(par ^ 1) * L + col] = v;
                }
            };
            if (chain) {
                T x = t_zero(T());
                unsigned long long key = 0ull;
                if (warp == 0 && c + 1 < L) {
                    // the next pivot column from the rows i > c, which nothing changes before the barrier below
                    if (lane < nloc && rank + C * lane > c)
                        x = t_fma(t_neg(f), pr[c + 1], M[(size_t)lane * LD + c + 1]);
                    x = search(c + 1, x, key);
                }
                asm volatile("bar.sync 1, %0;" ::"r"(kRhiThreads) : "memory");
                if (c + 1 < L) {
                    const int li = s_li;
                    if (warp == 0) {
                        publish(par ^ 1, x, key, li);
                    } else {
                        // the candidate row and row c + 1, updated and published
                        const int two = (li >= 0 ? 1 : 0) + (ln >= 0 && ln != li ? 1 : 0);
                        for (int t = warp - 1; t < two * nb; t += kRhiChain - 1)
                            update(t < nb && li >= 0 ? li : ln, t % nb, true);
                    }
                    cluster_arrive();
                }
                // row c becomes the scaled pivot row
                if (own_c) {
                    T* row = M + (size_t)((c - rank) / C) * LD;
                    for (int col = tid; col < L; col += 32 * kRhiChain) row[col] = col == c ? pinv : t_mul(pr[col], pinv);
                }
            } else {
                // items (row, column block), one warp each, in turn: rows i < c first, a
                // few of them while the chain warps search, the rest with the rows i > c
                const int b = warp < 8 ? warp - kRhiChain : warp - kRhiChain - 1;
                const bool work = warp != 8;
                int li = b / nb, cb = b % nb;
                if (work) {
                    for (int t = 0; t < kRhiEarly && li < done; ++t) {
                        update(li, cb, false);
                        for (cb += kRhiBulk; cb >= nb; cb -= nb) ++li;
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"r"(kRhiThreads) : "memory");
                if (c + 1 < L) cluster_arrive();
                const int li0 = c + 1 < L ? s_li : -1;
                const int nskip = (li0 >= 0 ? 1 : 0) + (ln >= 0 && ln != li0 ? 1 : 0);
                const int sa = li0 >= 0 && ln >= 0 ? min(li0, ln) : max(li0, ln), sb = max(li0, ln);
                if (work) {
                    const int nrows = nloc - (own_c ? 1 : 0) - nskip;   // all but row c and the chain's rows
                    while (li < nrows) {
                        int row = li < done ? li : li + (own_c ? 1 : 0);
                        if (nskip > 0 && row >= sa) ++row;
                        if (nskip > 1 && row >= sb) ++row;
                        update(row, cb, false);
                        for (cb += kRhiBulk; cb >= nb; cb -= nb) ++li;
                    }
                }
            }
        }
        if (!ok) break;
        __syncthreads();
        // S <- (S + S^{-1}) / 2 and the relative Frobenius change; the
        // interchanges are undone on the columns of the inverse
        int* pm = reinterpret_cast<int*>(prow);
        if (tid < L) pm[tid] = perm;
        __syncthreads();
        double dsum = 0.0, nsum = 0.0;
        for (int e = tid; e < nloc * L; e += blockDim.x) {
            int li = e / L, col = e % L;
            size_t gi = (size_t)(rank + C * li) * L + col;
            T so = S[gi];
            T sn = t_scale(t_add(so, M[(size_t)li * LD + pm[col]]), 0.5);
            dsum += t_norm2(t_sub(sn, so));
            nsum += t_norm2(sn);
            S[gi] = sn;
        }
        dsum = block_sum(dsum, sh1);
        nsum = block_sum(nsum, sh1);
        const int ip = it & 1;
        if (tid < C) {
            double* dst = cl.map_shared_rank(&part[ip][rank][0], tid);
            dst[0] = dsum;
            dst[1] = nsum;
        }
        cl.sync();
        double dt = 0.0, nt = 0.0;
        for (int q = 0; q < C; ++q) {
            dt += part[ip][q][0];
            nt += part[ip][q][1];
        }
        if (sqrt(dt) <= stop * sqrt(nt)) { converged = true; break; }
    }
    cl.sync();   // no CTA leaves while others read its buffers
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

static_assert(kRhiThreads >= 256, "one thread per column of the largest l");

template <typename T>
static size_t rhi_smem(int ell, int C) {
    int nmax = (ell + C - 1) / C;
    return (size_t)nmax * (ell + 1) * sizeof(T) + 6 * (size_t)ell * sizeof(T) + (size_t)nmax * sizeof(T);
}

static size_t rhi_smem_max() { return rhi_smem<double2>(256, 8); }

template <typename T>
static cudaError_t launch_rhi_t(const Inner& in, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kRhiThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto shape = [&](int C) {
        cfg.gridDim = dim3(in.n_rhs * C);
        cfg.dynamicSmemBytes = rhi_smem<T>(in.ell, C);
        attr[0].val.clusterDim.x = C;
    };
    int C = in.ell >= 64 ? 8 : (in.ell >= 16 ? 4 : 1);
    if (in.ell >= 96 && in.n_rhs <= 8) {
        // 16 CTAs (a size the device may not offer) halve the update of a large
        // matrix, while the chip holds the clusters of all RHS at once.  The inner part with
        // 8 -> 16 CTAs, ms: two-sided, k = 1024, l = 128: 1 RHS 7.62 -> 6.74, 7 7.66 -> 6.77,
        // 8 7.66 -> 7.57, 10 7.66 -> 7.79; k = 512, l = 256: 1 27.6 -> 17.0, 8 31.6 -> 26.8 (and
        // 12 43.2 -> 35.2); l = 96: 3.96 -> 3.97.  Hermitian: l = 256 1 12.7 -> 7.9, 8 14.5 -> 10.6;
        // l = 128 1 3.64 -> 3.62, 8 3.70 -> 3.82; l = 96 1 2.20 -> 2.30
        shape(16);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_rhi<T>, &cfg) == cudaSuccess && n > 0) C = 16;
        else cudaGetLastError();
    }
    shape(C);
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

// Test harness for the scalar helpers of the recurrences and of the inner part
// (nk_common.cuh, inner_arith.cuh).  Reads from stdin n, then n pairs (x, y); runs
// every helper on each and writes, per pair, 18 numbers: sqrt_inv(|x|) and its
// inverse; beta, gamma, 1 / beta, 1 / gamma of csqrt_scalars(x + i y); pivot_inv and
// pivot_div of x; pivot_inv and pivot_div of x + i y; step_scalars<false>(x).beta and its
// inverse.
#include <cstdio>
#include <vector>

#include "inner_arith.cuh"
#include "nk_step.cuh"

constexpr int kOut = 18;

__global__ void helpers(const double2* in, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 z = in[i];
    double* o = out + (size_t)i * kOut;
    o[0] = nk::sqrt_inv(fabs(z.x), o[1]);
    double2 b, g, ib, ig;
    nk::csqrt_scalars(z, b, g, ib, ig);
    o[2] = b.x; o[3] = b.y; o[4] = g.x; o[5] = g.y;
    o[6] = ib.x; o[7] = ib.y; o[8] = ig.x; o[9] = ig.y;
    o[10] = nk::pivot_inv(z.x);
    o[11] = nk::pivot_div(z.x);
    const double2 pi = nk::pivot_inv(z), pd = nk::pivot_div(z);
    o[12] = pi.x; o[13] = pi.y; o[14] = pd.x; o[15] = pd.y;
    const nk::StepScalars t = nk::step_scalars<false>(z);
    o[16] = t.beta.x;
    o[17] = t.ok ? t.inv_beta.x : -1.0;
}

int main() {
    int n;
    if (std::scanf("%d", &n) != 1 || n < 1) return 2;
    std::vector<double2> in(n);
    for (auto& z : in)
        if (std::scanf("%lf %lf", &z.x, &z.y) != 2) return 2;
    double2* din = nullptr;
    double* dout = nullptr;
    std::vector<double> out((size_t)n * kOut);
    if (cudaMalloc(&din, n * sizeof(double2)) != cudaSuccess || cudaMalloc(&dout, out.size() * sizeof(double)) != cudaSuccess ||
        cudaMemcpy(din, in.data(), n * sizeof(double2), cudaMemcpyHostToDevice) != cudaSuccess)
        return 3;
    helpers<<<(n + 127) / 128, 128>>>(din, dout, n);
    if (cudaMemcpy(out.data(), dout, out.size() * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    for (int i = 0; i < n; ++i)
        for (int c = 0; c < kOut; ++c) std::printf("%.17g%c", out[(size_t)i * kOut + c], c + 1 < kOut ? ' ' : '\n');
    return 0;
}

// Accuracy of the exponential that tree attention's softmax takes on the FMA pipe (ex2_pair_fma) and of ex2.approx.ftz.f32, which it
// takes for the rest, against exp2 in double: every fp32 in [-126, 127] whose bits differ in the top 19 (the exponent and 10 bits of
// the mantissa) with eight endings each, both places of the pair; then the values at and beyond the ends, infinities and NaN.
//
//   nvcc -gencode arch=compute_100a,code=sm_100a -O3 -std=c++17 -I ../csrc -I ../../include -o exp2_error exp2_error.cu && ./exp2_error
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "cb_tc_dev.cuh"

__global__ void k(const float* x, float* fma, float* approx, int n) {
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (i + 1 >= n) return;
    ex2_pair_fma(f2_pack(x[i], x[i + 1]), fma[i], fma[i + 1]);
    approx[i] = ex2(x[i]);
    approx[i + 1] = ex2(x[i + 1]);
}

int main() {
    std::vector<float> x = {-INFINITY, -1e30f, -300.f, -127.5f, -127.f, -126.5f, 127.f, 127.01f, 300.f, INFINITY, NAN, 0.f};
    const int n_edge = (int)x.size();
    for (uint32_t hi = 0; hi < 1u << 19; ++hi)
        for (uint32_t lo = 0; lo < 8; ++lo) {
            const uint32_t bits = hi << 13 | lo * 1170u;
            float v;
            std::memcpy(&v, &bits, 4);
            if (v >= -126.f && v <= 127.f) x.push_back(v);
        }
    if (x.size() & 1) x.push_back(0.25f);
    const int n = (int)x.size();
    float *dx, *df, *da;
    if (cudaMalloc(&dx, 4ull * n) || cudaMalloc(&df, 4ull * n) || cudaMalloc(&da, 4ull * n)) return 1;
    cudaMemcpy(dx, x.data(), 4ull * n, cudaMemcpyHostToDevice);
    k<<<(n / 2 + 255) / 256, 256>>>(dx, df, da, n);
    std::vector<float> f(n), a(n);
    cudaMemcpy(f.data(), df, 4ull * n, cudaMemcpyDeviceToHost);
    if (cudaMemcpy(a.data(), da, 4ull * n, cudaMemcpyDeviceToHost) != cudaSuccess) { printf("%s\n", cudaGetErrorString(cudaGetLastError())); return 1; }
    double ef = 0, ea = 0, sf = 0;
    for (int i = n_edge; i < n; ++i) {
        const double t = std::exp2((double)x[i]), rf = f[i] / t - 1.0, ra = a[i] / t - 1.0;
        ef = std::fmax(ef, std::fabs(rf));
        if (t >= 1.1754943508222875e-38) ea = std::fmax(ea, std::fabs(ra));   // the smallest normal number: below it ex2.approx.ftz gives zero
        sf += rf;
    }
    printf("values %d\nfma_max_rel %.3e\nfma_mean_rel %.3e\napprox_max_rel %.3e\n", n - n_edge, ef, sf / (n - n_edge), ea);
    for (int i = 0; i < n_edge; ++i) printf("edge %g %.17g %.17g\n", x[i], f[i], a[i]);
    return 0;
}

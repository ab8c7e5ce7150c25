// The covariance's digit path when its waits run out: a limit of 200 cycles ends every
// wait for a first copy.  The kernel must return (all copies landed, tensor memory
// freed) with NaN in every entry that the digits give, the FP64 entries (column 70) as
// ever, and the next call with the usual limit must be right.
// tests/test_gpu_covariance_wait.py compiles and runs it.
#include <cmath>
#include <cstdio>
#include <vector>

#include "../../paper_1708_05303_gb300/csrc/bsp_cov.cu"

bsp_status bsp::record_cuda_error(cudaError_t, const char*) { return BSP_ECUDA; }

int main() {
    const int m = 700, d = 300, direct = 70;
    std::vector<double> x((size_t)m * d), c((size_t)d * d), ref((size_t)d * d);
    unsigned s = 1;
    for (double& v : x) v = ((s = s * 1664525u + 1013904223u) >> 8) * 0x1p-24 - 0.25;
    for (int k = 0; k < m; ++k) x[(size_t)k * d + direct] *= 1e150;
    double *dx, *mean, *cov;
    void* ws;
    const size_t wb = bsp::cov_layout(m, d).end;
    if (cudaMalloc(&dx, x.size() * 8) || cudaMalloc(&mean, d * 8) || cudaMalloc(&cov, c.size() * 8) || cudaMalloc(&ws, wb)) return 2;
    cudaMemcpy(dx, x.data(), x.size() * 8, cudaMemcpyHostToDevice);
    if (bsp_covariance(m, d, dx, mean, cov, 0) != BSP_OK) return 3;
    cudaMemcpy(ref.data(), cov, ref.size() * 8, cudaMemcpyDeviceToHost);
    for (long long wlim : {bsp::WAIT_CYCLES, 200ll, bsp::WAIT_CYCLES}) {
        cudaMemset(cov, 0, c.size() * 8);
        if (bsp::launch_cov_digits(m, d, dx, mean, cov, ws, wlim, 0) != cudaSuccess) return 4;
        if (cudaDeviceSynchronize() != cudaSuccess) return 5;
        cudaMemcpy(c.data(), cov, c.size() * 8, cudaMemcpyDeviceToHost);
        int nan = 0, bad = 0;
        for (int i = 0; i < d; ++i)
            for (int j = 0; j < d; ++j) {
                const double v = c[(size_t)i * d + j], r = ref[(size_t)i * d + j];
                const double tol = 1e-12 * std::sqrt(ref[(size_t)i * d + i]) * std::sqrt(ref[(size_t)j * d + j]);
                if (std::isnan(v)) ++nan;
                else if (!(std::fabs(v - r) <= tol)) ++bad;
            }
        std::printf("limit %lld: %d NaN, %d wrong\n", wlim, nan, bad);
        if (bad || nan != (wlim == 200 ? (d - 1) * (d - 1) : 0)) return 1;
    }
    return 0;
}

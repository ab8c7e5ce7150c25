// The contraction's error word: the first wait of a thread block that gives up records its
// bit, the waits that its abort then stops add none.  tests/test_gpu_error_word.py runs it.
#include <cstdio>

#include "../../paper_1708_05303_gb300/csrc/bsp_tc.cu"

bsp_status bsp::record_cuda_error(cudaError_t, const char*) { return BSP_ECUDA; }

__global__ void probe(bsp::TcSmem* s, int* err) {
    bsp::set_abort(s[0], err, 8);
    bsp::set_abort(s[0], err, 64);
    bsp::set_abort(s[0], err, 1);
    bsp::set_abort(s[1], err + 1, 64);   // another block's
}

int main() {
    bsp::TcSmem* s;
    int *err, host[2];
    if (cudaMalloc(&s, 2 * sizeof(bsp::TcSmem)) || cudaMalloc(&err, 8) || cudaMemset(s, 0, 2 * sizeof(bsp::TcSmem)) || cudaMemset(err, 0, 8)) return 2;
    probe<<<1, 1>>>(s, err);
    if (cudaMemcpy(host, err, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    std::printf("%d %d\n", host[0], host[1]);
    return !(host[0] == 8 && host[1] == 64);
}

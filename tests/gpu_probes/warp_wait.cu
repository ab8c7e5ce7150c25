// The pipelines' bounded wait (bsp_ptx.h, warp_wait): true where every lane's barrier is
// complete, false where one is open until the limit or an abort, and the same in every
// lane.  One warp; barriers that nothing completes stand for a wait that never ends; every
// wait here is bounded by its limit or by an abort flag that is already set.
// tests/test_gpu_warp_wait.py runs it.
#include <cstdio>

#include "../../paper_1708_05303_gb300/csrc/bsp_ptx.h"

using namespace bsp;

__global__ void probe(int* out) {
    __shared__ uint64_t done, open;
    __shared__ volatile int abort;
    const int lane = threadIdx.x;
    if (lane == 0) {
        mbar_init(&done, 1);
        mbar_init(&open, 1);
        abort = 0;
        mbar_arrive(&done);   // phase 0 of this one completes
    }
    __syncwarp();
    const uint32_t d = smem_u32(&done), o = smem_u32(&open), mixed = lane < 31 ? d : o;
    int r[11];
    r[0] = warp_wait<1>(d, 0, 1000, &abort);
    r[1] = warp_wait<1>(o, 0, 1000, &abort);              // polls until the limit
    r[2] = warp_wait<64>(mixed, 0, 5000, &abort);         // one lane's barrier is open
    r[3] = warp_wait<1>(o, 0, 1ll << 21, &abort);         // sleeps until the limit (about 1 ms)
    __syncwarp();
    abort = 1;
    __syncwarp();
    r[4] = warp_wait<1>(o, 0, WAIT_CYCLES, &abort);
    r[5] = warp_wait<64>(mixed, 0, WAIT_CYCLES, &abort);
    r[6] = warp_wait<1>(d, 0, WAIT_CYCLES, &abort);       // complete all the same
    r[9] = warp_wait<1>(mixed, 0, 1ll << 21, nullptr);    // nothing but the limit ends this one
    r[10] = warp_wait<1>(d, 0, 300, nullptr);
    __syncwarp();
    abort = 0;
    __syncwarp();
    r[7] = warp_wait<1>(o, 0, 300, &abort);
    r[8] = warp_wait<1>(d, 0, 300, &abort);
    for (int i = 0; i < 11; ++i) out[i * 32 + lane] = r[i];
}

int main() {
    int *dev, host[11 * 32];
    if (cudaMalloc(&dev, sizeof(host))) return 2;
    probe<<<1, 32>>>(dev);
    if (cudaMemcpy(host, dev, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    const int want[11] = {1, 0, 0, 0, 0, 0, 1, 0, 1, 0, 1};
    int bad = 0;
    for (int i = 0; i < 11; ++i)
        for (int l = 0; l < 32; ++l)
            if (host[i * 32 + l] != want[i]) std::printf("wait %d lane %d: %d\n", i, l, host[i * 32 + l]), ++bad;
    return bad != 0;
}

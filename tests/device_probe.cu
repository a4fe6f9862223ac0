// Kernels that run single device functions of the library, for tests (built by device_probe.py).
#include "../paper_1605_01715_gb300/csrc/pair_tc.cuh"

using namespace kifmm;

namespace {

// One warp on a fresh barrier: a wait for parity 1 passes at once, one for parity 0 never
// does and ends by the abort flag.
__global__ void k_wait_warp(const int* parity, int raised, int* got) {
    __shared__ uint64_t bar;
    __shared__ int flag;
    if (threadIdx.x == 0) {
        flag = raised;
        tc::mbar_init(&bar, 1);
    }
    __syncwarp();
    got[threadIdx.x] = tc::mbar_wait_warp(&bar, (uint32_t)parity[threadIdx.x], &flag);
}

}  // namespace

// parity, got: 32 ints on the device.
extern "C" int probe_wait_warp(const int* parity, int raised, int* got) {
    k_wait_warp<<<1, 32>>>(parity, raised, got);
    cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}

// Kernels that run single device functions of the library, for tests (built by device_probe.py).
#include "../paper_1605_01715_gb300/csrc/pair_tc.cuh"
#include "../paper_1605_01715_gb300/csrc/sliced.cuh"

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

// The sliced products' parameters: slices, bits of a vector's fixed point, pairs a tile.
extern "C" void probe_slice_params(int* out) {
    out[0] = kSlices;
    out[1] = kSliceBits;
    out[2] = kSlicePairs;
}

// slice_eval_rows of n targets (all arrays on the device; slices: n x slice_cols(Q) x kSlices FP16).
extern "C" int probe_eval_rows(const int* tleaf_of, int n, const double* txyz, const double* tnrm, int axis, const int* lvl,
                               const double* ctr, double root_h, const double* bpts, int Q, int grad, void* slices, int* exps,
                               double* oscale) {
    KF_TRY(slice_eval_rows(tleaf_of, 0, n, n, txyz, tnrm, axis, lvl, ctr, root_h, bpts, Q, grad != 0, (__half*)slices, exps,
                           oscale, 0));
    return cudaDeviceSynchronize() == cudaSuccess ? KIFMM_OK : KIFMM_ERR_CUDA;
}

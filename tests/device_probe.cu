// Kernels that run single device functions of the library, for tests (built by device_probe.py).
#include "../paper_1605_01715_gb300/csrc/pair_tc.cuh"
#include "../paper_1605_01715_gb300/csrc/plan.cuh"
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

// Slices the operators (nops of Mr rows x K, row stride ld) and vectors (nvec, stride vld),
// both on the device, and multiplies the tiles' pairs (tiles: 4 ints each, on the host): added
// into the doubles out, or with oscale stored as floats.
extern "C" int probe_sliced_product(const double* table, int nops, int Mr, int K, int ld, int M, const double* vec, int nvec,
                                    int vld, const int* tiles, int ntiles, const int* pin, const int* pout, void* out,
                                    int ostride, const double* oscale, int* err) {
    SlicedTable t;
    DBuf<__half> sl;
    DBuf<int> ex;
    DBuf<int4> dt;
    std::vector<int4> ht(ntiles);
    for (int i = 0; i < ntiles; ++i) ht[i] = make_int4(tiles[4 * i], tiles[4 * i + 1], tiles[4 * i + 2], tiles[4 * i + 3]);
    KF_TRY(slice_table(table, nops, Mr, K, ld, t, 0));
    KF_TRY(sl.alloc((size_t)nvec * slice_cols(K) * kSlices));
    KF_TRY(ex.alloc(nvec));
    KF_TRY(dt.upload(ht, 0));
    KF_TRY(slice_vectors(vec, K, vld, 0, nvec, sl.p, ex.p, 0));
    if (oscale)
        KF_TRY(launch_sliced_store<float>(t, M, dt.p, ntiles, pin, pout, sl.p, ex.p, oscale, (float*)out, ostride, err, 0));
    else
        KF_TRY(launch_sliced_add(t, M, dt.p, ntiles, pin, pout, sl.p, ex.p, (double*)out, ostride, err, 0));
    return cudaDeviceSynchronize() == cudaSuccess ? KIFMM_OK : KIFMM_ERR_CUDA;
}

extern "C" int probe_chain_early(int captured, int kernel, long long near_pairs, int x_list, long long units,
                                 long long resident) {
    return chain_early(captured != 0, kernel, near_pairs, x_list != 0, units, resident);
}

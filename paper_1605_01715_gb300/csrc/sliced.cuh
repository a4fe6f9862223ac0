// FP64 products on the tensor cores from exact FP16 slices (the error-free splitting of
// matrix products of Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59, 2012).
//
// A vector with |x| < 2^e is rounded once to the fixed point of 62 bits, x = 2^(e - 62) n:
// exact for entries down to 2^-9 of the largest.  n is written in balanced base-128 digits
// n = sum_s digit_s 128^(8 - s), digit_s in [-64, 64]: nine FP16 slices of small integers.  A
// product of two vectors is then a sum over slice pairs (i, j) of integer dot products.  Those
// with i + j <= 8 are kept, summed by d = i + j: for d <= 7 at most 8 pairs x 512 columns x 2^12 =
// 2^24, so FP32 accumulators of the tensor core hold them exactly, whatever it does to bits below
// its last place.  (The last, of 9 pairs, could pass 2^24 and lose a unit or two an MMA, 2^-68 of
// the largest products each: far below what is left out.)  The accumulators are combined in
// 64-bit integers and two FP64 terms.
//
// Error per column, for |a| < 2^ea and |b| < 2^eb: 2^-62 of 2^(ea + eb) from the fixed point,
// and at most 1.008 x 2^-60 from the pairs left out (eight with i + j = 9 of 2^12 x 128^7 each,
// over 2^124); each entry may be 2^(e - 1), so 2^-57.7 of the product of the largest entries.
// FP64 products err by 2^-53 of each term and of each partial sum.  On the method's own
// operators and check potentials (p = 3 to 10, all families) the error is at most 0.4 of that of
// FP64 FMAs in order.  Eight slices with i + j <= 7 (at most 2^-51 per column) made up to 22 times
// that error, where a row's largest entries meet the vector's smallest: neighbouring boxes of
// the double layer at p = 6.  45 FP16 slice products in place of FP64 FMAs (2 per clock and SM here).
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace kifmm {

constexpr int kSlices = 9;
constexpr int kSliceBits = 7 * kSlices - 1;   // of the fixed point: the largest entry is below 2^kSliceBits
constexpr int kSlicePairs = 48;         // columns (pairs) per tile
constexpr int kSliceRows = 128;         // operator rows per work item

// Columns of a sliced vector: K rounded up to the 32 of a pipeline stage.
inline int slice_cols(int K) { return (K + 31) / 32 * 32; }

// Sliced operator tables: plane s holds digit s of every row (op * Mr + row), slice_cols(K)
// wide, rows scaled by 2^(kSliceBits - exp); map: its TMA map over all planes.
struct SlicedTable {
    DBuf<__half> planes;
    DBuf<int> exp;
    CUtensorMap map;
    int Mr = 0, K = 0;
    int64_t rows = 0;                   // of one plane
    size_t bytes() const { return planes.bytes() + exp.bytes(); }
};

// Slice a row-major FP64 table of nops operators of Mr rows x K columns (row stride ld).
int slice_table(const double* table, int64_t nops, int Mr, int K, int ld, SlicedTable& t, cudaStream_t s);

// Slice vectors v[b][0..K) (stride ld) for b in [b0, b1): slices[b] holds slice_cols(K) x 9
// FP16 as [block of 32 columns][slice][32]; exps[b] = e (kNotFinite if an entry is not
// finite: its products are NaN).
constexpr int kNotFinite = -100000;
int slice_vectors(const double* v, int K, int ld, int b0, int b1, __half* slices, int* exps, cudaStream_t s);

// out[pout[j]][row] (+)= sum_k Op[row][k] in[pin[j]][k] for every pair of the tiles (op,
// first pair, pairs <= kSlicePairs, 0), rows < M.  FP64: added by atomics into ostride
// doubles per output.  FP32 store: written, times oscale[pout[j]], with zeros in
// rows M..ostride.  err: a word a wait that gave up sets.
int launch_sliced_add(const SlicedTable& t, int M, const int4* tiles, int ntiles, const int* pin, const int* pout,
                      const __half* in, const int* exps, double* out, int ostride, int* err, cudaStream_t s);
template <typename Real>
int launch_sliced_store(const SlicedTable& t, int M, const int4* tiles, int ntiles, const int* pin, const int* pout,
                        const __half* in, const int* exps, const double* oscale, Real* out, int ostride,
                        int* err, cudaStream_t s);

// Evaluation rows of targets [t0, t0 + n): for target t of leaf b, at x in the leaf's unit
// frame, the Q values 1/|x - b_m| or (grad) nvec . (x - b_m)/|x - b_m|^3, nvec the target
// normal tnrm or the unit vector of coordinate axis, as the sliced vectors slices[t - t0]
// (exps), and oscale[t - t0] = 1 or (grad) 1 / half-width of the leaf.
int slice_eval_rows(const int* tleaf_of, int64_t t0, int n, int64_t nt, const double* txyz, const double* tnrm, int axis,
                    const int* lvl, const double* ctr, double root_h, const double* bpts, int Q, bool grad,
                    __half* slices, int* exps, double* oscale, cudaStream_t s);

// Digits of y (|y| <= 2^62) in balanced base 128, most significant first.
__device__ __forceinline__ void slice_digits(long long y, __half* d) {
#pragma unroll
    for (int s = kSlices - 1; s > 0; --s) {
        const int r = (int)((y + 64) & 127) - 64;
        d[s] = __int2half_rn(r);
        y = (y - r) >> 7;
    }
    d[0] = __int2half_rn((int)y);
}

// e with |x| < 2^e for the largest magnitude m (0 for m = 0; m finite).
__device__ __forceinline__ int slice_exp(double m) { return m > 0.0 ? ilogb(m) + 1 : 0; }

}  // namespace kifmm

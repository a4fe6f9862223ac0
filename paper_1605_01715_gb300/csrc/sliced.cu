// FP64 products from exact FP16 slices on the tensor cores (see sliced.cuh): slicing, the
// persistent tcgen05 kernel and its launchers.
#include <cmath>
#include <type_traits>

#include "sliced.cuh"
#include "pair_tc.cuh"

namespace kifmm {

int tc_make_map_rows(CUtensorMap* map, const __half* p, int64_t nrows, int Kp, int box_rows);

namespace {

using namespace tc;

constexpr int kOzStages = 2;                                  // ring depth
constexpr int kOzABytes = kSliceRows * (int)kRowBytes;        // one slice of the operator rows, one stage
constexpr int kOzBBytes = kSlicePairs * (int)kRowBytes;       // one slice of the inputs, one stage
constexpr int kOzStageBytes = kSlices * (kOzABytes + kOzBBytes);
constexpr int kOzSmemBytes = kOzStages * kOzStageBytes + 1024;
constexpr int kOzChunk = 16;                                  // stages accumulators 0 to 7 stay exact over: 512 columns
constexpr int kOzWarps = 12, kOzThreads = kOzWarps * 32;
constexpr int kOzProdWarp0 = 2, kOzProdThreads = 64;
constexpr int kOzFoldWarp0 = 4, kOzFoldThreads = 256;
constexpr int kOzFoldCols = kSlicePairs / 2;                  // columns of a fold warp
static_assert(kSlices == 9 && kOzFoldCols % 8 == 0 && kSlicePairs % 16 == 0, "the copies' and folds' shares");
static_assert(kOzStageBytes % 1024 == 0 && kOzSmemBytes <= 227 * 1024, "two stages fit");
static_assert(kSlices * kSlicePairs <= 512, "one accumulator per digit sum fits TMEM");
static_assert((long long)(kSlices - 1) * 64 * 64 * kOzChunk * kKS <= 1LL << 24, "all accumulators but the last stay exact");
static_assert(kOzBBytes % 512 == 0 && kSlicePairs % 16 == 0, "slices of the inputs follow one another as rows of one operand");

// x 2^e
__device__ __forceinline__ double scale2(double x, int e) {
    if (e < -1000 || e > 1000) return scalbn(x, e);
    return x * __longlong_as_double((long long)(1023 + e) << 52);
}

// One warp per vector: largest magnitude, then the digits.  PLANES: an operator table
// (plane-major); else a box vector ([32-column block][slice][32]).
template <bool PLANES>
__global__ void __launch_bounds__(256) k_slice(const double* __restrict__ v, int K, int Kc, int ld, int64_t b0, int64_t b1,
                                               int64_t plane, __half* __restrict__ out, int* __restrict__ exps) {
    const int lane = threadIdx.x & 31;
    const int64_t b = b0 + blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
    if (b >= b1) return;
    const double* x = v + (size_t)b * ld;
    double m = 0.0;
    bool fin = true;
    for (int k = lane; k < K; k += 32) {
        const double a = fabs(x[k]);
        fin = fin && isfinite(a);
        m = fmax(m, a);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    fin = __all_sync(0xffffffffu, fin);
    const int e = fin ? slice_exp(m) : 0;
    if (lane == 0) exps[b] = fin ? e : kNotFinite;
    for (int k = lane; k < Kc; k += 32) {
        __half d[kSlices];
        slice_digits(fin && k < K ? __double2ll_rn(scale2(x[k], kSliceBits - e)) : 0LL, d);
#pragma unroll
        for (int s = 0; s < kSlices; ++s) {
            if (PLANES) out[(size_t)s * plane + (size_t)b * Kc + k] = d[s];
            else out[((size_t)b * Kc + (k & ~31)) * kSlices + s * 32 + (k & 31)] = d[s];
        }
    }
}

// Nearest integer to x 2^(kSliceBits - e) (halves away from zero) for finite |x| < 2^e, from
// x's own bits: the conversion would take the FP64 pipe.
__device__ __forceinline__ long long fixed_point(double x, int e) {
    const long long u = __double_as_longlong(x);
    const int ex = (int)((u >> 52) & 0x7ff);
    if (ex == 0) return x == 0.0 ? 0LL : __double2ll_rn(scalbn(x, kSliceBits - e));      // subnormal
    const long long m = (u & 0xfffffffffffffLL) | 0x10000000000000LL;       // x = m 2^(ex - 1075)
    const int sh = ex - 1075 + kSliceBits - e;                              // at most 9
    long long y = sh >= 0 ? m << sh : (sh > -64 ? ((m >> (-sh - 1)) + 1) >> 1 : 0LL);
    return u < 0 ? -y : y;
}

// One warp per target, NV kernel values a lane.
template <int NV>
__global__ void __launch_bounds__(128) k_slice_eval(const int* __restrict__ tleaf_of, int64_t t0, int n, int64_t nt,
                                                    const double* __restrict__ txyz, const double* __restrict__ tnrm,
                                                    int axis, const int* __restrict__ lvl, const double* __restrict__ ctr,
                                                    double root_h, const double* __restrict__ bpts, int Q, int Kc,
                                                    bool grad, __half* __restrict__ out, int* __restrict__ exps,
                                                    double* __restrict__ oscale) {
    const int lane = threadIdx.x & 31, i = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (i >= n) return;
    const int64_t t = t0 + i;
    const int b = tleaf_of[t];
    const double r = ldexp(root_h, -lvl[b]);
    double x[3], nv[3];
    for (int d = 0; d < 3; ++d) {
        x[d] = (txyz[d * nt + t] - ctr[3 * b + d]) / r;
        nv[d] = tnrm ? tnrm[d * nt + t] : (d == axis ? 1.0 : 0.0);
    }
    double v[NV];
    int top = 0;                                  // largest exponent field
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int k = j * 32 + lane;
        v[j] = 0.0;
        if (k < Q) {
            const double dx = x[0] - bpts[3 * k], dy = x[1] - bpts[3 * k + 1], dz = x[2] - bpts[3 * k + 2];
            const double inv = rsqrt(dx * dx + dy * dy + dz * dz);
            v[j] = grad ? (nv[0] * dx + nv[1] * dy + nv[2] * dz) * (inv * inv * inv) : inv;
        }
        top = max(top, (__double2hiint(v[j]) >> 20) & 0x7ff);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    const bool fin = top < 0x7ff;
    const int e = fin ? top - 1022 : 0;           // |v| < 2^e
    if (lane == 0) {
        exps[i] = fin ? e : kNotFinite;
        oscale[i] = grad ? 1.0 / r : 1.0;
    }
    __half* o = out + (size_t)i * Kc * kSlices + lane;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        if (j * 32 >= Kc) break;
        __half d[kSlices];
        slice_digits(fin ? fixed_point(v[j], e) : 0LL, d);
#pragma unroll
        for (int s = 0; s < kSlices; ++s) o[(size_t)j * 32 * kSlices + s * 32] = d[s];
    }
}

// The nine digit sums (integers in FP32) as one double, sum_d acc_d 128^-d: two
// 64-bit integers below 2^51, each made a double by placing it in the mantissa of a number
// whose last place has its weight (2^-28, 2^-56), and one add.  Three FP64 adds in all.
__device__ __forceinline__ double join_digits(const uint32_t (&v)[kSlices][8], int c) {
    static_assert(kSlices == 9, "digits 0 to 4 and 5 to 8");
    long long h = 0, l = 0;
#pragma unroll
    for (int d = 0; d < 5; ++d) h = h * 128 + __float2int_rn(__uint_as_float(v[d][c]));
#pragma unroll
    for (int d = 5; d < 9; ++d) l = l * 128 + __float2int_rn(__uint_as_float(v[d][c]));
    const double ch = 0x1.8p24, cl = 0x1.8p-4;
    return (__longlong_as_double(__double_as_longlong(ch) + h) - ch) + (__longlong_as_double(__double_as_longlong(cl) + l) - cl);
}

// STORE: write Real(oscale * value) (zeros in rows M .. ostride); else add into doubles.
// Persistent over items (tile, group of 128 rows).  Warp 0: TMA of the operator slices;
// warp 1: the MMAs of a stage (45 slice products x 2 K steps in 26 MMAs of 48 to 240 columns),
// issued by an elected lane; warps 2-3: cp.async of the gathered input slices; warps 4-11: digit
// sums to FP64 and out.
// What bounds it: a stage takes 3.7 k clk with its share of the joins, 27 B a clock and SM of its
// 99 KB of operands, the L2 fabric's rate as in the translation kernel; its MMAs are 2.2 k at the
// tensor core's rate (one MMA a slice product would read A 45 times a K step instead of 13).  Tiles are 48 columns wide because nine
// accumulators fill tensor memory's 512.  Joining the digit sums (three FP64 adds and a product
// per output) is not overlapped.
// 46,080-point sphere at p = 12 (K = 728, 80,360 V pairs): M2L 89.0 ms in FP64 FMAs, 3.44 with
// eight slices in narrow MMAs, 3.08 so; U2U and L2L 29.9, 0.29 and 0.23 ms each.  Evaluation rows of
// 98,000 targets at p = 10 (with their slicing): 21.7, 2.9 and 2.8 ms.
template <typename Real, bool STORE>
__global__ void __launch_bounds__(kOzThreads, 1)
k_sliced(const __grid_constant__ CUtensorMap map, int64_t plane_rows, const int* __restrict__ aexp, int M, int Mr,
         int Kc, int mgroups, int nitems, const int4* __restrict__ tiles, const int* __restrict__ pin,
         const int* __restrict__ pout, const __half* __restrict__ in, const int* __restrict__ bexp,
         const double* __restrict__ oscale, Real* __restrict__ out, int ostride, int* __restrict__ err) {
    const int G = gridDim.x;
    const int K = nitems > (int)blockIdx.x ? (nitems - (int)blockIdx.x + G - 1) / G : 0;
    if (K == 0) return;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    __shared__ uint64_t tma_full[kOzStages], b_full[kOzStages], empty[kOzStages];
    __shared__ uint64_t acc_full, acc_empty, drain_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int nst = Kc / kKS;
    volatile int* abort = &s_abort;
    auto item = [&](int k) { return (int)blockIdx.x + k * G; };
    auto stage = [&](int s) -> uint32_t { return base + (uint32_t)(s * kOzStageBytes); };
    if (tid == 0) {
        s_abort = 0;
        for (int i = 0; i < kOzStages; ++i) {
            mbar_init(&tma_full[i], 1);
            mbar_init(&b_full[i], kOzProdThreads);
            mbar_init(&empty[i], 1);
        }
        mbar_init(&acc_full, 1);
        mbar_init(&acc_empty, kOzFoldThreads);
        mbar_init(&drain_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        // ---- operator slices by TMA ----
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int k = 0; k < K && ok; ++k) {
                const int arow = tiles[item(k) / mgroups].x * Mr + (item(k) % mgroups) * kSliceRows;
                for (int i = 0; i < nst; ++i, ++g) {
                    const int s = g % kOzStages;
                    if (g >= kOzStages && !mbar_wait_ab(&empty[s], (uint32_t)(((g / kOzStages) - 1) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&tma_full[s], (uint32_t)(kSlices * kOzABytes));
                    for (int d = 0; d < kSlices; ++d)
                        tma_load_2d(stage(s) + (uint32_t)(d * kOzABytes), &map, i * kKS, (int)(d * plane_rows) + arow,
                                    &tma_full[s]);
                }
            }
            // every issued load has landed before the CTA can end
            for (int s = 0; s < kOzStages && s < g; ++s) {
                const int last = s + ((g - 1 - s) / kOzStages) * kOzStages;
                if (!mbar_wait(&tma_full[s], (uint32_t)((last / kOzStages) & 1))) *abort = 1;
            }
        }
    } else if (warp == 1) {
        // ---- MMA issue: slice pairs (i, j) with i + j <= 8 into accumulator i + j.  Slices j
        // of the inputs follow one another in shared memory and accumulators i + j in tensor
        // memory, so slice i of the operator takes its 9 - i partners in one or two wide MMAs ----
        const bool leader = elect_one();
        const uint64_t d0 = smem_desc(stage(0));
        bool ok = true;
        int g = 0, f = 0;
        for (int k = 0; k < K && ok; ++k)
            for (int i0 = 0; i0 < nst && ok; i0 += kOzChunk, ++f) {
                const int i1 = i0 + kOzChunk < nst ? i0 + kOzChunk : nst;
                bool got = f == 0 || mbar_wait_ab(&acc_empty, (uint32_t)((f - 1) & 1), abort);
                for (int i = i0; i < i1; ++i, ++g) {
                    const int s = g % kOzStages;
                    const uint32_t ph = (uint32_t)((g / kOzStages) & 1);
                    got = got && mbar_wait_ab(&tma_full[s], ph, abort) && mbar_wait_ab(&b_full[s], ph, abort);
                    if (!__all_sync(0xffffffffu, got)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    if (leader) {
                        const uint64_t a0 = d0 + (uint32_t)s * (kOzStageBytes >> 4);
                        const uint64_t b0 = a0 + ((kSlices * kOzABytes) >> 4);
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                            for (int a = 0; a < kSlices; ++a) {
                                const int nb = kSlices - a, w = nb > 5 ? (nb + 1) / 2 : nb;   // N <= 256
#pragma unroll
                                for (int b = 0; b < nb; b += w)
                                    mma_f16(tmem + (uint32_t)((a + b) * kSlicePairs), a0 + a * (kOzABytes >> 4) + ks * 2,
                                            b0 + b * (kOzBBytes >> 4) + ks * 2,
                                            idesc_f16(128, (b + w < nb ? w : nb - b) * kSlicePairs),
                                            (i == i0 && ks == 0 && a == 0) ? 0u : 1u);
                            }
                        mma_commit(&empty[s]);
                        if (i == i1 - 1) mma_commit(&acc_full);
                    }
                    __syncwarp();
                }
            }
        if (g > 0) {
            if (leader) mma_commit(&drain_bar);
            __syncwarp();
            if (!mbar_wait(&drain_bar, 0)) *abort = 1;
        }
    } else if (warp < kOzFoldWarp0) {
        // ---- input slices by cp.async: a pair's 32 columns are 9 slices x 64 B in a row, 36
        // chunks of 16 bytes.  Warp w copies pairs w, w + 2, ...: a chunk a lane of slices 0 to 7
        // of one pair after the other, and slice 8 of eight pairs at a time ----
        const int r0 = warp - kOzProdWarp0, cc = lane & 3, u = lane >> 2;
        int g = 0;
        bool ok = true;
        for (int k = 0; k < K && ok; ++k) {
            const int4 t = tiles[item(k) / mgroups];
            // lane l holds the boxes of pairs r0 + 2 l
            const int r = r0 + 2 * lane;
            const int mine = r < t.z ? pin[t.y + r] : -1;
            for (int i = 0; i < nst; ++i, ++g) {
                const int s = g % kOzStages;
                const bool got = g < kOzStages || mbar_wait_ab(&empty[s], (uint32_t)(((g / kOzStages) - 1) & 1), abort);
                if (!__all_sync(0xffffffffu, got)) {
                    ok = false;
                    break;
                }
                const uint32_t bs = stage(s) + (uint32_t)(kSlices * kOzABytes);
                auto copy = [&](int m, int slice) {        // this lane's chunk of the m-th pair's slice
                    const int bi = __shfl_sync(0xffffffffu, mine, m);
                    const __half* src = in + ((size_t)(bi < 0 ? 0 : bi) * Kc + i * kKS) * kSlices + slice * 32 + cc * 8;
                    cp_async16(bs + (uint32_t)(slice * kOzBBytes) + sw64_off(r0 + 2 * m, cc), src, bi < 0 ? 0u : 16u);
                };
#pragma unroll
                for (int m0 = 0; m0 < kSlicePairs / 2; m0 += 8) {
#pragma unroll
                    for (int m = m0; m < m0 + 8; ++m) copy(m, u);
                    copy(m0 + u, 8);
                }
                cp_async_commit();
                // the copies have landed before the next stage's begin: two stages hide it
                cp_async_wait<0>();
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(&b_full[s]);
            }
        }
    } else {
        // ---- digit sums to FP64: lane quarter warp % 4, columns 24 half .. + 23 ----
        const int quarter = warp & 3, half = (warp - kOzFoldWarp0) >> 2;
        const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * kOzFoldCols);
        int f = 0;
        for (int k = 0; k < K; ++k) {
            const int4 t = tiles[item(k) / mgroups];
            const int row = (item(k) % mgroups) * kSliceRows + quarter * 32 + lane;
            const int re = row < M ? aexp[(size_t)t.x * Mr + row] - 12 : 0;
            double sum[kOzFoldCols];
#pragma unroll
            for (int j = 0; j < kOzFoldCols; ++j) sum[j] = 0.0;
            bool ok = true;
            for (int i0 = 0; i0 < nst; i0 += kOzChunk, ++f) {
                if (!mbar_wait_warp(&acc_full, (uint32_t)(f & 1), abort)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < kOzFoldCols; c0 += 8) {
                    uint32_t v[kSlices][8];
#pragma unroll
                    for (int d = 0; d < kSlices; ++d) tmem_ld<8>(ta + (uint32_t)(d * kSlicePairs + c0), v[d]);
                    tmem_wait_ld();
                    if (c0 + 8 == kOzFoldCols) {
                        tc_fence_before();
                        mbar_arrive(&acc_empty);
                    }
#pragma unroll
                    for (int c = 0; c < 8; ++c) sum[c0 + c] += join_digits(v, c);
                }
            }
            if (!ok) break;
            if (row < (STORE ? ostride : M)) {
#pragma unroll
                for (int j = 0; j < kOzFoldCols; ++j) {
                    const int col = half * kOzFoldCols + j;
                    if (col >= t.z) break;
                    const int ob = pout[t.y + col];
                    const int be = bexp[pin[t.y + col]];
                    const double x = be == kNotFinite ? __longlong_as_double(0x7ff8000000000000LL) : scale2(sum[j], re + be);
                    if constexpr (STORE) out[(size_t)ob * ostride + row] = (Real)(row < M ? x * oscale[ob] : 0.0);
                    else atomicAdd(out + (size_t)ob * ostride + row, x);
                }
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort) atomicOr(err, 1);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

template <typename Real, bool STORE>
int launch(const SlicedTable& t, int M, const int4* tiles, int ntiles, const int* pin, const int* pout,
           const __half* in, const int* bexp, const double* oscale, Real* out, int ostride, int* err,
           cudaStream_t s) {
    if (ntiles <= 0) return KIFMM_OK;
    auto kern = k_sliced<Real, STORE>;
    KF_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kOzSmemBytes));
    int dev = 0, nsm = 0;
    KF_CHECK_CUDA(cudaGetDevice(&dev));
    KF_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int mgroups = ((STORE ? std::max(M, ostride) : M) + kSliceRows - 1) / kSliceRows;
    const int nitems = ntiles * mgroups;
    kern<<<nitems < nsm ? nitems : nsm, kOzThreads, kOzSmemBytes, s>>>(t.map, t.rows, t.exp.p, M, t.Mr, slice_cols(t.K),
                                                                       mgroups, nitems, tiles, pin, pout, in, bexp,
                                                                       oscale, out, ostride, err);
    KF_CHECK_LAUNCH();
    return KIFMM_OK;
}

}  // namespace

int slice_table(const double* table, int64_t nops, int Mr, int K, int ld, SlicedTable& t, cudaStream_t s) {
    const int Kc = slice_cols(K);
    t.Mr = Mr;
    t.K = K;
    t.rows = nops * Mr;
    KF_TRY(t.planes.alloc((size_t)kSlices * t.rows * Kc));
    KF_TRY(t.exp.alloc((size_t)t.rows));
    k_slice<true><<<(unsigned)((t.rows + 7) / 8), 256, 0, s>>>(table, K, Kc, ld, 0, t.rows, t.rows * Kc, t.planes.p, t.exp.p);
    KF_CHECK_LAUNCH();
    return tc_make_map_rows(&t.map, t.planes.p, kSlices * t.rows, Kc, kSliceRows);
}

int slice_vectors(const double* v, int K, int ld, int b0, int b1, __half* slices, int* exps, cudaStream_t s) {
    if (b1 <= b0) return KIFMM_OK;
    k_slice<false><<<(b1 - b0 + 7) / 8, 256, 0, s>>>(v, K, slice_cols(K), ld, b0, b1, 0, slices, exps);
    KF_CHECK_LAUNCH();
    return KIFMM_OK;
}

int slice_eval_rows(const int* tleaf_of, int64_t t0, int n, int64_t nt, const double* txyz, const double* tnrm, int axis,
                    const int* lvl, const double* ctr, double root_h, const double* bpts, int Q, bool grad,
                    __half* slices, int* exps, double* oscale, cudaStream_t s) {
    if (n <= 0) return KIFMM_OK;
    auto kern = Q <= 320 ? k_slice_eval<10> : Q <= 640 ? k_slice_eval<20> : k_slice_eval<43>;
    kern<<<(n + 3) / 4, 128, 0, s>>>(tleaf_of, t0, n, nt, txyz, tnrm, axis, lvl, ctr, root_h, bpts, Q, slice_cols(Q), grad,
                                     slices, exps, oscale);
    KF_CHECK_LAUNCH();
    return KIFMM_OK;
}

int launch_sliced_add(const SlicedTable& t, int M, const int4* tiles, int ntiles, const int* pin, const int* pout,
                      const __half* in, const int* bexp, double* out, int ostride, int* err, cudaStream_t s) {
    return launch<double, false>(t, M, tiles, ntiles, pin, pout, in, bexp, nullptr, out, ostride, err, s);
}

template <typename Real>
int launch_sliced_store(const SlicedTable& t, int M, const int4* tiles, int ntiles, const int* pin, const int* pout,
                        const __half* in, const int* bexp, const double* oscale, Real* out, int ostride,
                        int* err, cudaStream_t s) {
    return launch<Real, true>(t, M, tiles, ntiles, pin, pout, in, bexp, oscale, out, ostride, err, s);
}
template int launch_sliced_store<float>(const SlicedTable&, int, const int4*, int, const int*, const int*, const __half*,
                                        const int*, const double*, float*, int, int*, cudaStream_t);

}  // namespace kifmm

// Grouped translation GEMM on the 5th-generation tensor cores (tcgen05), two-term FP16.
//
// A work item is one tile of up to N (input box, output box) pairs that share one
// operator Op (Mr x Kp rows and columns of a table of such operators: a translation,
// or a projection onto a check-space basis) and one group of 128 * SLABS rows:
//   out[pout[j]][row] += sum_k Op[row][k] * in[pin[j]][k]
// computed as D(128 x N) = A(128 x K) B(N x K)^T per 128-row slab, with A = operator
// rows and B = the gathered input vectors, accumulated in TMEM.
//
// Two-term FP16: every operand is scaled by a power of two into [2^14, 2^15) at its
// largest entry and written as x = x_hi + x_lo with x_hi, x_lo the nearest FP16 values
// (22 significant bits); D += A_hi B_hi + A_hi B_lo + A_lo B_hi (the dropped A_lo B_lo
// term is ~2^-22 relative) with kind::f16 MMAs, and the epilogue undoes both scales.
// Operator tables have one scale each (texp); input vectors one per box (bexp), and
// both come pre-split: the operators once at setup, the box vectors right before the
// launch (one pass over the input buffer).
//
// Accumulation: the tensor core adds into its FP32 accumulator with truncation, so a
// long K loop into one accumulator drifts by ~1 ulp of the running sum per MMA.  Every
// stage (32 columns of K) therefore starts a fresh accumulator (correction products first,
// then the hi*hi products), and the fold warps add each into FP32 registers
// (round-to-nearest).  The truncation dominates the rounding error of the whole
// mixed-precision matvec: folding every 32 columns instead of every 64 halved it (1M-point
// cube at p = 10, sampled rel-L2 8.9e-7 -> 4.4e-7).
//
// Schedule: persistent, one CTA per SM walking the items blockIdx.x + k * gridDim.x.  An
// item has two halves of 128 rows x 128 columns, each with its own accumulator, and the
// warps are split into roles joined only by mbarriers, so that the MMAs, the folds and the
// scatter of an item all run beside one another:
//   warps 0-1   MMA issue, one warp a half: while one waits, the other's MMAs run
//   warps 2-3   operands: TMA of the operator rows, cp.async of the input rows, straight
//               into the layout
//   warps 4-11  fold of each accumulator into registers, four warps a half; the item's
//               finished sums are parked in the other 256 TMEM columns
//   warps 12-15 scatter of the parked sums (FP32 reds of four rows) beside the next item
// over a ring of kStages K-stages of 32 columns in the canonical K-major 64-byte-swizzled
// layout (rows of 64 B, 16-byte chunks XOR-permuted by row within 512-byte atoms).
// What bounds it: a stage's 12 MMAs take 830 clk and the operand loads and the scatter of
// all SMs keep the L2 fabric at about 10 TB/s, 1800 clk a stage.  1M-point sphere (975,296
// pairs, K = 302) 726 -> 494 us, 64-sphere pack (925,240, K = 256) 584 -> 391 us, 1M-point
// cube (271,952, chained) 186 -> 129 us against folds and scatter in one team of warps.
// A tile of few pairs works on its columns only (rounded to 16).
// Every wait is bounded; a wait that runs out raises an abort flag that stops the other
// roles, each of which then waits (bounded) for its own copies or MMAs in flight; the CTA
// records the error, frees its TMEM and returns.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace kifmm {
namespace tc {

constexpr int kKS = 32;                 // K elements (FP16) per ring stage: 2 MMA k-steps of 16
constexpr int kStages = 4;              // ring depth
constexpr int kBLag = 1;                // stages of input copies a producer thread keeps in flight (2: a
                                        // stage's MMAs then wait for the ring to turn, 4 % slower)
static_assert(kBLag < kStages, "ring too shallow for the copy lag");
constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kProdWarp0 = 2, kProdThreads = 64;     // operand loads
constexpr int kFoldWarp0 = 4, kFoldThreads = 256;    // folds of the accumulators
constexpr int kScatWarp0 = 12, kScatThreads = 128;   // scatter of the finished sums
constexpr int kPartThreads = kFoldThreads / 2;       // fold threads of one half of an item
constexpr int kFoldBar = 1, kScatBar = 2;            // named barriers of those roles
constexpr uint32_t kRowBytes = kKS * 2;              // 64 B: one swizzle row
constexpr uint32_t kSBO = 8 * kRowBytes;             // 512 B between 8-row groups
constexpr int kSlabBytes = 128 * kRowBytes;          // one 128-row slab of one stage: 8 KB
constexpr int kScaleTop = 14;                        // operands scaled into [2^14, 2^15)
// Registers a thread: the block is launched with kLaunchRegs for each of its threads (all
// of the SM's, checked before each launch), and the other warps hand theirs to the fold
// warps, which hold 128 sums and 64 loaded columns each.  The shares may not exceed what
// the block was launched with.
constexpr int kLaunchRegs = 128, kProdRegs = 40, kFoldRegs = 208, kScatRegs = 56;
static_assert(kFoldWarp0 % 4 == 0 && kScatWarp0 % 4 == 0 && kProdRegs % 8 == 0 && kFoldRegs % 8 == 0 && kScatRegs % 8 == 0 &&
                  32 * (kFoldWarp0 * kProdRegs + (kScatWarp0 - kFoldWarp0) * kFoldRegs +
                        (kWarps - kScatWarp0) * kScatRegs) <= kThreads * kLaunchRegs,
              "register split within the launch's registers");
static_assert(kRowBytes == 64, "the 64-byte swizzle needs 32 FP16 per row");
static_assert(kFoldThreads == (kScatWarp0 - kFoldWarp0) * 32 && kProdThreads == (kFoldWarp0 - kProdWarp0) * 32 &&
                  kScatThreads == (kWarps - kScatWarp0) * 32,
              "role split");
constexpr long long kSpinLimit = 1LL << 26;

// Tile shape: SLABS x 128 operator rows by N pairs, in two halves of 128 rows x 128 columns
// (the slabs of <2, 128>, the column halves of <1, 256>).  Each half has one accumulator
// of 128 TMEM columns -- the MMAs of one half run while the other's is folded -- and the
// finished sums of both are parked in the other 256 columns for the scatter.
template <int SLABS, int N>
struct Shape {
    static constexpr int kRows = SLABS * 128;
    static constexpr int kTmemCols = 512;
    static constexpr int kPark = 256;                          // first column of the parked sums
    static constexpr int kABytes = SLABS * kSlabBytes;        // per hi or lo table, one stage
    static constexpr int kBBytes = N * (int)kRowBytes;         // per hi or lo table, one stage
    static constexpr int kStageBytes = 2 * kABytes + 2 * kBBytes;
    static constexpr int kSmemBytes = kStages * kStageBytes + 1024;
    static constexpr int kBRows = N / 16;                      // input rows per producer thread
    static_assert(SLABS * N == 256, "two halves of 128 x 128");
    static_assert(kStageBytes % 1024 == 0, "stages stay 1024-byte aligned");
    // operator row (within the item) and column where half p starts
    __host__ __device__ static constexpr int row(int p) { return SLABS == 2 ? p * 128 : 0; }
    __host__ __device__ static constexpr int col(int p) { return SLABS == 2 ? 0 : p * 128; }
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// K-major, 64-byte swizzle: 8-row groups kSBO apart, leading offset unused (1),
// descriptor version 1, layout type 4 (SWIZZLE_64B).  Tiles are 1024-byte aligned; a K
// step of 16 inside the 64-byte row advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((kSBO >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// 2-D tiled TMA load of one box into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// kind::f16 instruction descriptor: D FP32, A/B FP16, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait; returns false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    for (long long i = 0; i < kSpinLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (i > 64) __nanosleep(64);
    }
    return false;
}

// Bounded wait that also gives up once another role has raised *abort; a timeout
// raises it.  Returns false if it gave up.
__device__ __forceinline__ bool mbar_wait_ab(uint64_t* bar, uint32_t parity, volatile int* abort) {
    for (long long i = 0; i < kSpinLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort) return false;
        if (i > 64) __nanosleep(32);
    }
    *abort = 1;
    return false;
}

// The same for a whole warp that goes on to warp-wide (.aligned) instructions.  Lanes that
// watch the barrier and *abort on their own can part, some passing and others giving up, when
// the barrier completes as the flag is raised: here each try is the warp's.  (A vote after
// lanes had waited on their own cost a 1M-point cube 0.2 %, 270,000 points 0.3 %; this does not.)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort) {
    for (long long i = 0; i < kSpinLimit; ++i) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if (__any_sync(0xffffffffu, *abort != 0)) return false;
        if (i > 64) __nanosleep(32);
    }
    *abort = 1;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Named barrier over the n threads of one role (id 0 is __syncthreads); the second
// form also returns whether pred held in any of them.
__device__ __forceinline__ void bar_named(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ bool bar_named_or(int id, int n, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %2, 0;\n\t"
        "bar.red.or.pred q, %1, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(id), "r"((uint32_t)pred), "r"(n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// One lane of the converged warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r));
    return r != 0;
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// COLS consecutive TMEM columns of the warp's 32 lanes into registers (one column each).
template <int COLS>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r) {
    static_assert(COLS == 8 || COLS == 16 || COLS == 32 || COLS == 64, "one load instruction");
#define KF_R8(o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
    if constexpr (COLS == 8) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];" : KF_R8(0) : "r"(taddr));
    } else if constexpr (COLS == 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
            "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
            : KF_R8(0), KF_R8(8)
            : "r"(taddr));
    } else if constexpr (COLS == 32) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
            "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
            "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
            : KF_R8(0), KF_R8(8), KF_R8(16), KF_R8(24)
            : "r"(taddr));
    } else {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
            "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
            "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
            "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
            "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];"
            : KF_R8(0), KF_R8(8), KF_R8(16), KF_R8(24), KF_R8(32), KF_R8(40), KF_R8(48), KF_R8(56)
            : "r"(taddr));
    }
#undef KF_R8
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// COLS registers into consecutive TMEM columns of the warp's 32 lanes.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float2* v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
#define KF_W4(o) "f"(v[o].x), "f"(v[o].y), "f"(v[o + 1].x), "f"(v[o + 1].y)
        KF_W4(0), KF_W4(2), KF_W4(4), KF_W4(6), KF_W4(8), KF_W4(10), KF_W4(12), KF_W4(14)
#undef KF_W4
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Adds COLS loaded columns of an accumulator into acc (COLS / 2 pairs), scaled per column
// when SCALED (osc: the columns' scales).  Packed FP32x2: the roundings of scalar adds.
template <int COLS, bool SCALED>
__device__ __forceinline__ void fold_add(const uint32_t* v, const float4* osc, float2* acc) {
#pragma unroll
    for (int j = 0; j < COLS; j += 4) {
        const float2 a = make_float2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
        const float2 b = make_float2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        if (SCALED) {
            const float4 sc = osc[j >> 2];
            acc[j >> 1] = __ffma2_rn(a, make_float2(sc.x, sc.y), acc[j >> 1]);
            acc[(j >> 1) + 1] = __ffma2_rn(b, make_float2(sc.z, sc.w), acc[(j >> 1) + 1]);
        } else {
            acc[j >> 1] = __fadd2_rn(a, acc[j >> 1]);
            acc[(j >> 1) + 1] = __fadd2_rn(b, acc[(j >> 1) + 1]);
        }
    }
}

// The first ncol (at most 128) columns, as few and as wide loads as cover them: each load
// and its wait are a serial step of the fold (eight 16-column loads took 1500 clk a stage,
// two of 64 take 480).  Columns past ncol that a load covers hold leftovers; their sums
// are never written.  free() is called once the last column is in registers.
template <bool SCALED, typename Free>
__device__ __forceinline__ void fold_acc(uint32_t taddr, int ncol, const float4* osc, float2* acc, Free free) {
    if (ncol > 32) {
        uint32_t v[64];
        tmem_ld<64>(taddr, v);
        tmem_wait_ld();
        if (ncol > 64) {
            fold_add<64, SCALED>(v, osc, acc);
            tmem_ld<64>(taddr + 64, v);
            tmem_wait_ld();
            free();
            fold_add<64, SCALED>(v, osc + 16, acc + 32);
        } else {
            free();
            fold_add<64, SCALED>(v, osc, acc);
        }
    } else if (ncol > 16) {
        uint32_t v[32];
        tmem_ld<32>(taddr, v);
        tmem_wait_ld();
        free();
        fold_add<32, SCALED>(v, osc, acc);
    } else if (ncol > 0) {
        uint32_t v[16];
        tmem_ld<16>(taddr, v);
        tmem_wait_ld();
        free();
        fold_add<16, SCALED>(v, osc, acc);
    } else {
        free();
    }
}

// B 4 x 4 transposes across each quad of lanes: lane l's v[4 b + c], the value of row l in
// column c, becomes the value of row c of the quad in column l & 3.
template <int B>
__device__ __forceinline__ void transpose4(int lane, uint32_t* v) {
    const bool b0 = lane & 1, b1 = lane & 2;
    uint32_t r[2 * B];
#pragma unroll
    for (int i = 0; i < 2 * B; ++i) r[i] = __shfl_xor_sync(0xffffffffu, b0 ? v[2 * i] : v[2 * i + 1], 1);
#pragma unroll
    for (int i = 0; i < 2 * B; ++i) {
        v[2 * i] = b0 ? r[i] : v[2 * i];
        v[2 * i + 1] = b0 ? v[2 * i + 1] : r[i];
    }
#pragma unroll
    for (int i = 0; i < 2 * B; ++i) {
        const int a = 4 * (i >> 1) + (i & 1);
        r[i] = __shfl_xor_sync(0xffffffffu, b1 ? v[a] : v[a + 2], 2);
    }
#pragma unroll
    for (int i = 0; i < 2 * B; ++i) {
        const int a = 4 * (i >> 1) + (i & 1);
        v[a] = b1 ? r[i] : v[a];
        v[a + 2] = b1 ? v[a + 2] : r[i];
    }
}

// Four consecutive floats added at p (16-byte aligned) where on.
__device__ __forceinline__ void red_add4(float* p, bool on, float a, float b, float c, float d) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "@p red.global.add.v4.f32 [%0], {%2, %3, %4, %5};\n\t}" ::"l"(p),
        "r"((uint32_t)on), "f"(a), "f"(b), "f"(c), "f"(d)
        : "memory");
}

// 2^e as a float (e in [-126, 127]).
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros and reads nothing.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

// Byte offset of (row r, 16-byte chunk c) in a K-major 64-byte-swizzled tile: the chunk
// index is XORed with bits 7-8 of the row's byte offset.
__device__ __forceinline__ uint32_t sw64_off(int r, int c) {
    return (uint32_t)(r * kRowBytes + ((c ^ ((r >> 1) & 3)) << 4));
}

// Columns of a tile of cnt pairs that the MMAs, the input copies, the folds and the scatter
// work on: cnt rounded up to the MMA's step of 16.
__host__ __device__ constexpr int tile_cols(int cnt) { return cnt <= 16 ? 16 : (cnt + 15) / 16 * 16; }
// Columns of half p of the item at row0 (0: none of the operator's M rows or the tile's
// columns fall in it).
template <int SLABS, int N>
__device__ __forceinline__ int half_cols(int p, int M, int row0, int cols) {
    if (SLABS == 2) return row0 + p * 128 < M ? cols : 0;
    return cols > p * 128 ? (cols - p * 128 < 128 ? cols - p * 128 : 128) : 0;
}

// tiles[t] = (op, first pair, count, chain); work item w = (tile w / mgroups, row group
// w % mgroups).  chain = 1 (only with mgroups = 1): item w + gridDim.x, this CTA's next,
// has the same output box in every column and its products are added to this item's
// before they are written.  kcount (null: all items c + k G) holds each CTA's item count.  map_hi / map_lo: 2-D tensor maps of the split FP16 operator tables
// (scaled by 2^texp), rows = op * Mr + row (Mr rows per operator), columns Kp, box = 32
// columns x kRows rows, 64-byte swizzle.  in_hi / in_lo: the input vectors of all boxes
// scaled by 2^bexp[box] and split, Kp FP16 per box.  out: ostride floats per box, of
// which rows < M are written (and zeros added to the last rows below ostride).
template <int SLABS, int N>
__device__ __forceinline__ void pair_tc_body(const CUtensorMap& map_hi, const CUtensorMap& map_lo, int texp, int M,
                                             int Kp, int ostride, int Mr, int mgroups, int nitems,
                                             const int4* __restrict__ tiles,
                                             const int* __restrict__ pin, const int* __restrict__ pout,
                                             const int* __restrict__ bexp, const __half* __restrict__ in_hi,
                                             const __half* __restrict__ in_lo, float* __restrict__ out,
                                             int* __restrict__ err, const int* __restrict__ kcount) {
    using S = Shape<SLABS, N>;
    const int G = gridDim.x;
    // items of this CTA: every G-th from blockIdx.x, or the first kcount[blockIdx.x] of them
    const int K = kcount ? kcount[blockIdx.x]
                         : (nitems > (int)blockIdx.x ? (nitems - (int)blockIdx.x + G - 1) / G : 0);
    pdl_trigger();
    if (K == 0) return;                   // uniform: nothing allocated yet
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    __shared__ uint64_t tma_full[kStages];    // operator rows of a stage landed (TMA bytes)
    __shared__ uint64_t b_full[kStages];      // input rows of a stage landed (producer arrivals)
    __shared__ uint64_t empty[kStages];       // MMAs reading a stage done
    __shared__ uint64_t acc_full[2];          // accumulator of a half complete
    __shared__ uint64_t acc_empty[2];         // accumulator of a half folded
    __shared__ uint64_t park_full;            // an item's sums parked
    __shared__ uint64_t park_empty;           // parked sums read
    __shared__ uint64_t drain_bar[2];         // all MMAs of a half done
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float s_oscale[3][N];     // fold warps: output unscale per pair, of three items
    __shared__ __align__(16) int s_out[N];             // scatter warps: the item's output box and unscale per pair
    __shared__ __align__(16) float s_scale[N];
    __shared__ int s_abort;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // uniform across the warp
    const int nst = (Kp + kKS - 1) / kKS;                     // stages per item (tail zero-filled)
    volatile int* abort = &s_abort;
    auto stage_u32 = [&](int s) -> uint32_t { return smem_u32(base) + (uint32_t)(s * S::kStageBytes); };
    auto item = [&](int k) { return (int)blockIdx.x + k * G; };
    auto item_row = [&](int k) { return (item(k) % mgroups) * S::kRows; };

    if (tid == 0) {
        s_abort = 0;
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&tma_full[i], 1);
            mbar_init(&b_full[i], kProdThreads);
            mbar_init(&empty[i], 2);                // both halves' MMAs
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], kPartThreads);
            mbar_init(&drain_bar[i], 1);
        }
        mbar_init(&park_full, kFoldThreads);
        mbar_init(&park_empty, kScatThreads);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(S::kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp < kFoldWarp0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProdRegs));
        if (warp < 2) {
            // ---- MMA issue, warp p for half p: one warp's waits pass behind the other's MMAs
            // (one warp for both halves spent half of each stage waiting).  The whole warp walks
            // the loop and one elected lane issues, so that descriptors and addresses stay in
            // uniform registers, where the MMA reads them (issued by one diverged thread, 12
            // MMAs took 1000 clk whatever their N) ----
            const int p = warp;
            const bool leader = elect_one();
            const uint32_t d = tmem + (uint32_t)(p * 128);
            // stage 0's operand descriptors; other stages and K steps are offsets of the
            // address field (16-byte units)
            const uint64_t a0 = smem_desc(stage_u32(0) + (uint32_t)(S::row(p) * (int)kRowBytes));
            const uint64_t b0 = smem_desc(stage_u32(0) + (uint32_t)(2 * S::kABytes + S::col(p) * (int)kRowBytes));
            bool ok = true;
            int g = 0;
            int cnt = tiles[item(0) / mgroups].z;
            for (int k = 0; k < K && ok; ++k) {
                const int hc = __shfl_sync(0xffffffffu, half_cols<SLABS, N>(p, M, item_row(k), tile_cols(cnt)), 0);
                const uint32_t idesc = idesc_f16(128, hc);
                if (k + 1 < K) cnt = tiles[item(k + 1) / mgroups].z;   // read while this item runs
                for (int i = 0; i < nst; ++i, ++g) {
                    const int s = g % kStages;
                    const uint32_t ph = (uint32_t)((g / kStages) & 1);
                    const bool got = (g == 0 || mbar_wait_ab(&acc_empty[p], (uint32_t)((g - 1) & 1), abort)) &&
                                     mbar_wait_ab(&tma_full[s], ph, abort) && mbar_wait_ab(&b_full[s], ph, abort);
                    if (!__all_sync(0xffffffffu, got)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    if (leader) {
                        // a fresh accumulator: the small correction products first, then
                        // hi * hi (fewer truncating adds at the accumulator's full magnitude)
                        const uint64_t a_hi = a0 + (uint32_t)s * (S::kStageBytes >> 4), a_lo = a_hi + (S::kABytes >> 4);
                        const uint64_t b_hi = b0 + (uint32_t)s * (S::kStageBytes >> 4), b_lo = b_hi + (S::kBBytes >> 4);
                        if (hc > 0) {
#pragma unroll
                            for (int ks = 0; ks < kKS / 16; ++ks) {   // 16 FP16 along K inside the swizzled row
                                mma_f16(d, a_hi + ks * 2, b_lo + ks * 2, idesc, ks == 0 ? 0u : 1u);
                                mma_f16(d, a_lo + ks * 2, b_hi + ks * 2, idesc, 1u);
                            }
#pragma unroll
                            for (int ks = 0; ks < kKS / 16; ++ks)
                                mma_f16(d, a_hi + ks * 2, b_hi + ks * 2, idesc, 1u);
                        }
                        mma_commit(&acc_full[p]);
                        mma_commit(&empty[s]);
                    }
                    __syncwarp();
                }
            }
            // every MMA of this warp (and the arrivals it owes) is done before the CTA can end
            if (g > 0) {
                if (leader) mma_commit(&drain_bar[p]);
                __syncwarp();
                if (!mbar_wait(&drain_bar[p], 0)) *abort = 1;
            }
        } else {
            // ---- operands.  Operator rows by TMA, from the first thread.  Input rows by
            // cp.async: thread pt copies 16-byte chunk pt % 4 of rows pt / 4 + 16 j, so four
            // neighbouring threads read one 64-byte row slice.  (A TMA gather of four 64-byte
            // rows takes 42 clk of the TMA unit: 2700 a stage, against 1100 for these.) ----
            const int pt = tid - kProdWarp0 * 32, rr = pt >> 2, c = pt & 3;
            int bo[S::kBRows];                       // the rows' offsets in 16-byte chunks, or -1
            int g = 0;
            bool ok = true;
            for (int k = 0; k < K && ok; ++k) {
                const int4 t = tiles[item(k) / mgroups];
                const int nrow = tile_cols(t.z) >> 4, arow = t.x * Mr + item_row(k);
#pragma unroll
                for (int j = 0; j < S::kBRows; ++j) {
                    const int r = j * 16 + rr;
                    bo[j] = r < t.z ? pin[t.y + r] * (Kp >> 3) + c : -1;
                }
                for (int i = 0; i < nst; ++i, ++g) {
                    const int s = g % kStages;
                    if (g >= kStages && !mbar_wait_ab(&empty[s], (uint32_t)(((g / kStages) - 1) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    if (pt == 0) {
                        mbar_expect_tx(&tma_full[s], 2u * S::kABytes);
                        tma_load_2d(stage_u32(s), &map_hi, i * kKS, arow, &tma_full[s]);
                        tma_load_2d(stage_u32(s) + S::kABytes, &map_lo, i * kKS, arow, &tma_full[s]);
                    }
                    if (g == 0) pdl_wait();        // the inputs; the operator's first rows are on their way
                    const uint32_t bh = stage_u32(s) + 2 * S::kABytes;
                    const bool inside = i * kKS + 8 * c < Kp;   // an 8-group lies wholly inside or outside Kp
#pragma unroll
                    for (int j = 0; j < S::kBRows; ++j) {
                        if (j >= nrow) break;
                        const bool v = bo[j] >= 0 && inside;
                        const size_t off = v ? ((size_t)(uint32_t)bo[j] + i * (kKS / 8)) * 8 : 0;
                        const uint32_t o = sw64_off(j * 16 + rr, c);
                        cp_async16(bh + o, in_hi + off, v ? 16u : 0u);
                        cp_async16(bh + S::kBBytes + o, in_lo + off, v ? 16u : 0u);
                    }
                    cp_async_commit();
                    if (g >= kBLag) {
                        // stage g - kBLag: this thread's copies have landed; hand them to the
                        // tensor core's (async) proxy and arrive
                        cp_async_wait<kBLag>();
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        mbar_arrive(&b_full[(g - kBLag) % kStages]);
                    }
                }
            }
            cp_async_wait<0>();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (ok)
                for (int gg = g > kBLag ? g - kBLag : 0; gg < g; ++gg) mbar_arrive(&b_full[gg % kStages]);
            // every issued load has landed before the CTA can end (not cut short by an abort)
            if (pt == 0)
                for (int s = 0; s < kStages && s < g; ++s) {
                    const int last = s + ((g - 1 - s) / kStages) * kStages;
                    if (!mbar_wait(&tma_full[s], (uint32_t)((last / kStages) & 1))) *abort = 1;
                }
        }
    } else if (warp < kScatWarp0) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFoldRegs));
        pdl_wait();
        // ---- folds: half `half`, lane quarter warp % 4 (the TMEM lanes this warp may read) ----
        const int ft = tid - kFoldWarp0 * 32, half = (warp - kFoldWarp0) >> 2;
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        float2 acc[64];                       // columns 2j and 2j+1 of this thread's row
        // An item's column scales (used in chains) come from three dependent loads (tile, pin,
        // bexp).  Each is issued one step of the item before's folds ahead of its use, and
        // they are stored before the barrier that ends those folds.  Three buffers: the one
        // written for item k + 1 was last read in item k - 2, which every fold thread has
        // left by the barrier of item k - 1.
        static_assert(N <= kFoldThreads, "one table entry per fold thread");
        int4 tile = tiles[item(0) / mgroups];
        int4 tnext = K > 1 ? tiles[item(1) / mgroups] : make_int4(0, 0, 0, 0);
        auto scale_of = [&](int mbi) { return pow2f(-((mbi >= 0 ? bexp[mbi] : 0) + texp)); };
        if (ft < N) s_oscale[0][ft] = scale_of(ft < tile.z ? pin[tile.y + ft] : -1);
        bar_named(kFoldBar, kFoldThreads);
        int mb = 0, parked = 0;               // item k's table buffer: k mod 3; items parked so far
        // A chain: consecutive items of this CTA with the same output box in every column
        // (tile.w = 1: the next item of this CTA continues it).  Its sums stay in acc
        // across its items and are written once, after the last.  Each fold adds its
        // columns already unscaled (by powers of two, so the sums round as if unscaled
        // at the end); outside chains the scatter unscales.
        bool cont_prev = false;
        for (int k = 0; k < K; ++k) {
            const int mbn = mb == 2 ? 0 : mb + 1;
            const float4* osc4 = reinterpret_cast<const float4*>(s_oscale[mb] + S::col(half));
            const int4 tnn = k + 2 < K ? tiles[item(k + 2) / mgroups] : make_int4(0, 0, 0, 0);
            const bool cont = mgroups == 1 && tile.w != 0, chained = cont || cont_prev;
            // this warp's columns of the item (none when its rows lie past the operator's)
            const int row = item_row(k) + S::row(half) + (warp & 3) * 32;
            const int ncol = row < M ? half_cols<SLABS, N>(half, M, item_row(k), tile_cols(tile.z)) : 0;
            if (!cont_prev) {
#pragma unroll
                for (int j = 0; j < 64; ++j) acc[j] = make_float2(0.f, 0.f);
            }
            const int mbi = ft < tnext.z ? pin[tnext.y + ft] : -1;
            float msc = 1.f;
            bool ok = true;
            for (int j = 0; j < nst; ++j) {
                if (!mbar_wait_warp(&acc_full[half], (uint32_t)((k * nst + j) & 1), abort)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                auto free = [&]() {
                    tc_fence_before();
                    mbar_arrive(&acc_empty[half]);
                };
                const uint32_t col = tmem + lanes + (uint32_t)(half * 128);
                if (chained) fold_acc<true>(col, ncol, osc4, acc, free);
                else fold_acc<false>(col, ncol, osc4, acc, free);
                if (j == 0) msc = scale_of(mbi);
            }
            if (ft < N) s_oscale[mbn][ft] = msc;
            // hand the sums to the scatter warps, once those have read the item before's
            if (ok && !cont) {
                if (parked > 0) ok = mbar_wait_warp(&park_empty, (uint32_t)((parked - 1) & 1), abort);
                tc_fence_after();
                if (ok) {
                    const uint32_t pk = tmem + lanes + (uint32_t)(S::kPark + half * 128);
#pragma unroll
                    for (int j = 0; j < 128; j += 32) {
                        if (j >= ncol) break;
                        tmem_st32(pk + (uint32_t)j, acc + j / 2);
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(&park_full);
                }
                ++parked;
            }
            if (bar_named_or(kFoldBar, kFoldThreads, !ok)) break;   // uniform across the fold warps
            cont_prev = cont;
            tile = tnext;
            tnext = tnn;
            mb = mbn;
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kScatRegs));
        pdl_wait();
        // ---- scatter of the parked sums, beside the next item's MMAs and folds: lane quarter
        // warp % 4 of both halves; each column is one output box's 32 consecutive rows.
        // All SMs together scatter 16 to 19 B per clock and SM (the L2 fabric's rate, wider
        // reds or plain stores no faster), about the time an item's MMAs take, so in series
        // with them the scatter was 40 % of an item. ----
        const int st = tid - kScatWarp0 * 32;
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        int parked = 0;
        bool cont_prev = false;
        for (int k = 0; k < K; ++k) {
            const int4 tile = tiles[item(k) / mgroups];
            const bool cont = mgroups == 1 && tile.w != 0, chained = cont || cont_prev;
            cont_prev = cont;
            if (cont) continue;
            bar_named(kScatBar, kScatThreads);     // the last item's table is no longer read
            for (int j = st; j < N; j += kScatThreads) {
                const int bi = j < tile.z ? pin[tile.y + j] : -1;
                s_out[j] = j < tile.z ? pout[tile.y + j] : -1;
                s_scale[j] = chained ? 1.f : pow2f(-((bi >= 0 ? bexp[bi] : 0) + texp));
            }
            const bool ok = mbar_wait_ab(&park_full, (uint32_t)(parked & 1), abort);
            ++parked;
            if (bar_named_or(kScatBar, kScatThreads, !ok)) break;   // uniform across the scatter warps
            tc_fence_after();
            const int row0 = item_row(k), cols = tile_cols(tile.z);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int wrow = row0 + S::row(p) + (warp & 3) * 32;      // the warp's first row
                const int ncol = wrow < M ? half_cols<SLABS, N>(p, M, row0, cols) : 0;
                const bool edge = wrow + 32 > M, dead = wrow + lane >= M, live = wrow + (lane & ~3) < ostride;
                const int* so = s_out + S::col(p) + (lane & 3);
                const float* sc = s_scale + S::col(p) + (lane & 3);
                const uint32_t pk = tmem + lanes + (uint32_t)(S::kPark + p * 128);
                float* orow = out + wrow + (lane & ~3);
                for (int j0 = 0; j0 < ncol; j0 += 16) {
                    uint32_t v[16];
                    tmem_ld<16>(pk + (uint32_t)j0, v);
                    tmem_wait_ld();
                    if (edge) {                       // rows past the operator's: add zeros
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = dead ? 0u : v[j];
                    }
                    // all four blocks' boxes, scales and transposes before the first red: four
                    // independent chains, and no branch between them
                    int ob[4];
                    float x[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        ob[j] = so[j0 + 4 * j];
                        x[j] = sc[j0 + 4 * j];
                    }
                    transpose4<4>(lane, v);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        red_add4(orow + (int64_t)ob[j] * ostride, ob[j] >= 0 && live, __uint_as_float(v[4 * j]) * x[j],
                                 __uint_as_float(v[4 * j + 1]) * x[j], __uint_as_float(v[4 * j + 2]) * x[j],
                                 __uint_as_float(v[4 * j + 3]) * x[j]);
                    __syncwarp();
                }
            }
            tc_fence_before();
            mbar_arrive(&park_empty);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort) atomicOr(err, 1);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kTmemCols)
                     : "memory");
    }
}

// One kernel name per translation so profiles tell them apart.
#define KF_TC_KERNEL(NAME)                                                                                \
    template <int SLABS, int N>                                                                                 \
    __global__ void __launch_bounds__(kThreads, 1)                                                              \
        NAME(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo, int M,     \
             int Kp, int ostride, int Mr, int mgroups, int nitems, const int4* __restrict__ tiles,               \
             const int* __restrict__ pin, const int* __restrict__ pout, const int* __restrict__ bexp, int texp,  \
             const __half* __restrict__ in_hi, const __half* __restrict__ in_lo, float* __restrict__ out,        \
             int* __restrict__ err, const int* __restrict__ kcount) {                                            \
        pair_tc_body<SLABS, N>(map_hi, map_lo, texp, M, Kp, ostride, Mr, mgroups, nitems, tiles, pin, pout,      \
                               bexp, in_hi, in_lo, out, err, kcount);                                            \
    }
KF_TC_KERNEL(k_u2u_tc)
KF_TC_KERNEL(k_m2l_tc)
KF_TC_KERNEL(k_l2l_tc)
KF_TC_KERNEL(k_proj_tc)
#undef KF_TC_KERNEL

}  // namespace tc
}  // namespace kifmm

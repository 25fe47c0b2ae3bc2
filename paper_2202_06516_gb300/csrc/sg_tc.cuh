// BF16 GEMM on the 5th-generation tensor cores (tcgen05, accumulators in tensor memory) for the
// surrogate network: C[M x N] = sum_k A(m, k) B(n, k), each operand K-major (A[m][k], B[n][k])
// or MN-major (A[k][m], B[k][n]): the forward convolution Xcol W^T and, with a transposed
// weight copy, the data gradient dY W (both K-major), and the weight gradient dY^T Xcol (both
// MN-major, K = pixels).
//
// One CTA of 128 threads computes a 128 x BN tile. Its K-slices reach shared memory either as
// cp.async gathers by all threads (TMA = 0), in the 128-byte-swizzled K-major layout the tensor
// core reads (8-row atoms of 1 KB; the 16-byte chunk c of row r stored at chunk c ^ (r % 8)), or
// as tensor-map (TMA) boxes issued by thread 0 (TMA = 64 / 32: K-major slices of 64 or 32
// elements, 128- or 64-byte swizzle; TMA = 1: the weight gradient's MN-major blocks), STAGES
// slices in flight. Thread 0 issues the 128 x BN x 16 MMAs of each slice (kind::f16, BF16 in,
// FP32 accumulate into BN tensor-memory columns) and commits them to the slice's mbarrier,
// which frees the slice for the next load. The epilogue reads the accumulator lanes back with
// tcgen05.ld (warp w owns rows 32 w .. 32 w + 31), adds the bias, applies the leaky ReLU and
// stores FP32 or BF16. k_wgrad_rows computes weight gradients of rows of 64 pixels and more from
// staged input rows, and k_conv_march the forward convolutions and data gradients
// of wide rows with few channels from operand rows staged once (the nine taps as operands shifted
// by whole pixels inside them).
//
// Every wait on an mbarrier is polled by one thread with an iteration limit; on expiry the
// CTA sets *err, waits (bounded) for the MMAs it issued, frees its tensor memory and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "sg_gemm.cuh"

namespace lbm {
namespace sgtc {

constexpr int BM = 128, BK = 64, TC_THREADS = 128;
constexpr long long kWaitLimit = 1ll << 22;

__host__ __device__ constexpr int tmem_cols(int bn) {
    return bn <= 32 ? 32 : bn <= 64 ? 64 : bn <= 128 ? 128 : 256;
}

// elements of K per stage of a kernel variant: 64, or 32 for the 64-byte-swizzled K-major TMA
// variant (TMA = 32); the launch sizes shared memory with the same rule as the kernel
__host__ __device__ constexpr int slice_k(int tma) { return tma == 64 || tma == 32 ? tma : BK; }

// KS: elements of K per stage (slice_k of the variant)
template <int BN, int STAGES, bool BMN = false, int KS = BK>
struct TcShape {
    static_assert(BN % 16 == 0 && BN >= 16 && BN <= 256, "MMA N of kind::f16 at M = 128");
    static constexpr int A_BYTES = BM * KS * 2;  // 16 KB (8 KB when KS = 32)
    // MN-major slices are whole 64-element swizzle atoms wide along M or N
    static constexpr int B_BYTES = BMN ? (BN + 63) / 64 * 64 * KS * 2 : BN * KS * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    // 1 KB alignment slack for the swizzle atoms, then the stages, mbarriers and the TMEM slot
    static constexpr int RAW_BYTES = 1024 + STAGES * STAGE_BYTES + 8 * (2 * STAGES + 1) + 16;
    // at least enough shared memory that the CTAs resident on one SM never ask for more than
    // the 512 tensor-memory columns together (an allocation beyond them would wait)
    static constexpr int TMEM_CTAS = 512 / tmem_cols(BN);
    static constexpr int MIN_BYTES = 233472 / (TMEM_CTAS + 1) + 1;
    static constexpr int SMEM_BYTES = RAW_BYTES > MIN_BYTES ? RAW_BYTES : MIN_BYTES;
};

__device__ __forceinline__ uint32_t su32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptors as two words. The high word is a constant of the layout: bytes
// between 8-row (K-major) or 8-K (MN-major) groups, the fixed version, the swizzle. The low word holds
// the start address / 16, which advances by bytes / 16, and for MN-major operands the bytes between
// blocks of the swizzle's width along M or N (1, unused, for K-major ones). Precomputed words
// matter: one thread issues the MMAs, and building two 64-bit descriptors for each took about as
// long as the MMA (k_conv_march 57 -> 44 and 34 -> 23 us on the full-resolution layers).
//   K-major, 128-byte swizzle (64 channels per row): groups 1 KB apart; 64-byte (32): 512 B;
//   32-byte (16): 256 B. MN-major, 64-byte swizzle: groups 512 B, 32-wide blocks lbo apart;
//   128-byte swizzle: groups 1 KB, 64-wide blocks 8 KB apart.
// A start may lie on any whole row of the layout: the swizzle follows the absolute address.
//   Without swizzle the unit is a core matrix of 8 rows x 16 bytes (128 contiguous bytes): K-major,
//   groups = the next 8 rows and lbo = the next 8 K; MN-major (8 K rows of 8 M or N values),
//   groups = the next 8 M or N and lbo = the next 8 K.
enum Swizzle { SW_NONE = 0, SW128 = 2, SW64 = 4, SW32 = 6 };
__host__ __device__ constexpr uint32_t desc_hi(int group_bytes, Swizzle sw) {
    return (uint32_t)(group_bytes >> 4) | (1u << 14) | ((uint32_t)sw << 29);
}
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo_bytes = 16) {
    return ((saddr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, each K-major (0) or
// MN-major (1: the operand's transpose bit), M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn = 0, int b_mn = 0) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}

// poll one phase of an mbarrier; false when the iteration limit ran out
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (long long i = 0; i < kWaitLimit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                       uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %6, 0;\n"
        " mov.b64 da, {%1, %2};\n mov.b64 db, {%3, %4};\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(tmem),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
        : "memory");
}

// the mbarrier expects `bytes` more transaction bytes (one arrival)
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// tiled tensor copies global -> shared, completion counted on an mbarrier; coordinates are
// innermost first, out-of-range elements are zero-filled
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
        "{%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
        "{%2, %3}], [%4];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// 32 consecutive FP32 accumulator columns of the warp's 32 lanes (one row per thread)
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// 16 consecutive FP32 accumulator columns of the warp's 32 lanes
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// one K-slice of ROWS x 64 elements of a K-major operand into the swizzled layout; rows past
// nrows and k past ke are zero-filled
template <int ROWS>
__device__ __forceinline__ void load_slice(uint8_t* s, const __nv_bfloat16* g, int ld, int row0,
                                           int nrows, int k0, int ke, int kperiod = 0) {
    constexpr int CHUNKS = ROWS * (BK / 8);
#pragma unroll 4
    for (int i = threadIdx.x; i < CHUNKS; i += TC_THREADS) {
        const int r = i >> 3, c = i & 7;
        const bool ok = (row0 + r < nrows) && (k0 + c * 8 < ke);
        const int kc = kperiod ? (k0 + c * 8) % kperiod : k0 + c * 8;
        const __nv_bfloat16* src = ok ? g + (size_t)(row0 + r) * ld + kc : g;
        uint8_t* dst = s + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
        sg::cp_async16(dst, src, ok);
    }
}

// one K-slice of 64 (K) x ROWS (M or N) elements of an MN-major operand (row k of the stored
// matrix holds consecutive M or N indices) into the swizzled MN-major layout: element (mn, k) in
// block mn / 64, K-group k / 8 (1 KB apart), row k % 8, 16-byte chunk ((mn % 64) / 8) ^ (k % 8);
// positions past nrows or ke are zero-filled
template <int ROWS>
__device__ __forceinline__ void load_slice_mn(uint8_t* s, const __nv_bfloat16* g, int ld,
                                              int row0, int nrows, int k0, int ke) {
    constexpr int CPR = ROWS / 8;  // 16-byte chunks per stored row (ROWS % 8 == 0)
    constexpr int CHUNKS = BK * CPR;
#pragma unroll 4
    for (int i = threadIdx.x; i < CHUNKS; i += TC_THREADS) {
        const int k = i / CPR, c = i - k * CPR;
        const bool ok = (row0 + c * 8 < nrows) && (k0 + k < ke);
        const __nv_bfloat16* src = ok ? g + (size_t)(k0 + k) * ld + row0 + c * 8 : g;
        uint8_t* dst = s + (c >> 3) * (BK / 8 * 1024) + (k >> 3) * 1024 + (k & 7) * 128 +
                       (((c & 7) ^ (k & 7)) << 4);
        sg::cp_async16(dst, src, ok);
    }
}

// One K-slice of 128 rows (output pixels m0 ..) x 64 (K) of the gathered convolution operand
// (see sg::ConvGather), in the K-major swizzled layout of load_slice. Thread t always fills the
// 16-byte chunk column t % 8 of rows t / 8 + 16 j (j = 0..7), whose pixel coordinates it keeps
// in yx[j] (y | x << 16) and nn[j] (image index, -1 past M).
__device__ __forceinline__ void load_slice_conv(uint8_t* s, const sg::ConvGather& cv,
                                                const int* yx, const int* nn, int k0, int ke) {
    const int c = threadIdx.x & 7;
    const int k = k0 + c * 8;
    const bool kok = k < ke;
    const int tap = k >> cv.lc, ci = k & ((1 << cv.lc) - 1);
    const int dy = tap / 3 - 1, dx = tap - (tap / 3) * 3 - 1;
    const int h1 = cv.H >> cv.up1, w1 = cv.W >> cv.up1;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int r = (threadIdx.x >> 3) + 16 * j;
        const int y = (yx[j] & 0xFFFF) + dy, x = (yx[j] >> 16) + dx, n = nn[j];
        const bool ok = kok && n >= 0 && y >= 0 && y < cv.H && x >= 0 && x < cv.W;
        const __nv_bfloat16* src = cv.x1;
        if (ok) {
            if (ci < cv.C1)
                src = cv.x1 + ((((size_t)n * h1 + (y >> cv.up1)) * w1 + (x >> cv.up1)) * cv.C1 + ci);
            else
                src = cv.x2 + ((((size_t)n * cv.H + y) * cv.W + x) * cv.C2 + (ci - cv.C1));
        }
        uint8_t* dst = s + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
        sg::cp_async16(dst, src, ok);
    }
}

// One K-slice of 128 source pixels x 64 (K) of the data-gradient operand (see
// sg::DgradGather) in the K-major swizzled layout; rows as in load_slice_conv (yx, nn).
__device__ __forceinline__ void load_slice_dgrad(uint8_t* s, const sg::DgradGather& dg,
                                                 const int* yx, const int* nn, int k0, int ke) {
    const int c = threadIdx.x & 7;
    const int k = k0 + c * 8;
    const bool kok = k < ke;
    const int co = k & ((1 << dg.lco) - 1), t = k >> dg.lco;  // t = s * 9 + tap
    const int sub = t / 9, tap = t - sub * 9;
    const int dy = tap / 3 - 1, dx = tap - (tap / 3) * 3 - 1;
    const int oy = (sub >> 1) - dy, ox = (sub & 1) - dx;  // sub = 0 unless up1
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int r = (threadIdx.x >> 3) + 16 * j;
        const int y = ((yx[j] & 0xFFFF) << dg.up1) + oy, x = ((yx[j] >> 16) << dg.up1) + ox;
        const int n = nn[j];
        const bool ok = kok && n >= 0 && y >= 0 && y < dg.H && x >= 0 && x < dg.W;
        const __nv_bfloat16* src =
            ok ? dg.dy + ((((size_t)n * dg.H + y) * dg.W + x) << dg.lco) + co : dg.dy;
        uint8_t* dst = s + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
        sg::cp_async16(dst, src, ok);
    }
}

// One K-slice of 64 pixels (K) x 128 im2col columns (M: (tap, channel) of the gathered
// convolution operand) in the MN-major swizzled layout, as the A operand of the transposed
// weight gradient. Thread t always fills the 16-byte column chunk t % 16 (columns
// m0 + 8 (t % 16) ..), whose tap and channel it decodes once (tc, cc: ci | tap << 16, -1 past
// M); its pixels are k0 + t / 16 + 8 j (j = 0..7). H and W are powers of two.
__device__ __forceinline__ void load_slice_mn_conv_a(uint8_t* s, const sg::ConvGather& cv,
                                                     int tc, int k0, int ke) {
    const int c = threadIdx.x & 15;
    const int ci = tc & 0xFFFF, tap = tc >> 16;
    const int dy = tap / 3 - 1, dx = tap - (tap / 3) * 3 - 1;
    const int h1 = cv.H >> cv.up1, w1 = cv.W >> cv.up1;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int k = (threadIdx.x >> 4) + 8 * j;
        const int p = k0 + k;
        const int y = ((p >> cv.lw) & (cv.H - 1)) + dy, x = (p & (cv.W - 1)) + dx;
        const int n = p >> (cv.lw + cv.lh);
        const bool ok = tc >= 0 && p < ke && y >= 0 && y < cv.H && x >= 0 && x < cv.W;
        const __nv_bfloat16* src = cv.x1;
        if (ok) {
            if (ci < cv.C1)
                src = cv.x1 + ((((size_t)n * h1 + (y >> cv.up1)) * w1 + (x >> cv.up1)) * cv.C1 + ci);
            else
                src = cv.x2 + ((((size_t)n * cv.H + y) * cv.W + x) * cv.C2 + (ci - cv.C1));
        }
        uint8_t* dst = s + (c >> 3) * (BK / 8 * 1024) + (k >> 3) * 1024 + (k & 7) * 128 +
                       (((c & 7) ^ (k & 7)) << 4);
        sg::cp_async16(dst, src, ok);
    }
}

// Epilogue of one 128 x BN output tile whose FP32 accumulator sits in tensor-memory columns
// tacc .. tacc + BN - 1 (zero: no K slices, the result is 0). Warp `warp` (0 .. 3) reads
// accumulator lanes 32 warp .. 32 warp + 31 (rows m0 + 32 warp ..) and passes them through its
// own 32 x 32 staging block ep (rows 144 B apart), so that stores write whole row segments:
// 16-byte vectors when the output allows (no accumulation or split, aligned rows), else one
// column per lane; bias, leaky ReLU, BF16 or FP32 (accumulated, split at nsplit, or transposed)
// as the arguments say. zoff: the split-K partial's offset.
template <int BN>
__device__ __forceinline__ void epilogue_tile(const sg::GemmArgs& g, uint32_t tacc, float* ep,
                                              int warp, int lane, int m0, int n0, bool zero,
                                              size_t zoff) {
    // FP32 outputs may accumulate and may be split at column nsplit into two tensors; the
    // vector path then takes a 32-column chunk that lies on one side of the split
    const bool vec = g.Cb ? (!g.accumulate && g.ldc % 8 == 0 && ((uintptr_t)g.Cb & 15) == 0)
                          : (g.ldc % 4 == 0 && zoff % 4 == 0 && ((uintptr_t)g.Cf & 15) == 0 &&
                             (!g.Cf2 || (g.ldc2 % 4 == 0 && g.nsplit % 4 == 0 &&
                                         ((uintptr_t)g.Cf2 & 15) == 0)));
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 32) {
        if (n0 + c0 >= g.N) break;
        const int w = BN - c0 >= 32 ? 32 : 16;
        float v[32];
        const uint32_t ta = tacc + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
        if (zero) {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = 0.f;
        } else if (w == 32) {
            tc_ld32(ta, v);
        } else {
            tc_ld16(ta, v);
        }
        if (g.tout) {
            // transposed FP32 store: for each column, the warp's 32 rows are consecutive
            const int m = m0 + warp * 32 + lane;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int n = n0 + c0 + j;
                if (j >= w || n >= g.N || m >= g.M) continue;
                float* o = g.Cf + (size_t)n * g.ldc + m + zoff;
                *o = g.accumulate ? *o + v[j] : v[j];
            }
            continue;
        }
#pragma unroll
        for (int j = 0; j < 32; j += 4)
            if (j < w)
                *reinterpret_cast<float4*>(ep + lane * 36 + j) =
                    make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        __syncwarp();
        const bool one_side = !g.Cf2 || n0 + c0 + 32 <= g.nsplit || n0 + c0 >= g.nsplit;
        if (vec && w == 32 && n0 + c0 + 32 <= g.N && one_side) {
            if (g.Cb) {
                // lane: row it * 8 + lane / 4, columns 8 (lane % 4) .. + 7
                const int cc = 8 * (lane & 3), n = n0 + c0 + cc;
                float bn[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) bn[j] = g.bias ? g.bias[n + j] : 0.f;
#pragma unroll
                for (int it = 0; it < 4; ++it) {
                    const int r = it * 8 + (lane >> 2);
                    const int m = m0 + sg::row_pixel(warp * 32 + r, g.rperm);
                    if (m >= g.M) continue;
                    const float4 x0 = *reinterpret_cast<const float4*>(ep + r * 36 + cc);
                    const float4 x1 = *reinterpret_cast<const float4*>(ep + r * 36 + cc + 4);
                    float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
                    uint4 o;
                    __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        float a0 = x[j] + bn[j], a1 = x[j + 1] + bn[j + 1];
                        if (g.relu) {
                            a0 = fmaxf(a0, 0.1f * a0);
                            a1 = fmaxf(a1, 0.1f * a1);
                        }
                        oh[j / 2] = __floats2bfloat162_rn(a0, a1);
                    }
                    *reinterpret_cast<uint4*>(g.Cb + (size_t)m * g.ldc + n) = o;
                }
            } else {
                // lane: row it * 4 + lane / 8, columns 4 (lane % 8) .. + 3
                const int cc = 4 * (lane & 7), n = n0 + c0 + cc;
                float bn[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) bn[j] = g.bias ? g.bias[n + j] : 0.f;
                // destination of row it * 4 + lane / 8; with accumulation all eight old
                // values are loaded before the first store, so their latencies overlap
                auto dst_of = [&](int it) {
                    const int m = m0 + sg::row_pixel(warp * 32 + it * 4 + (lane >> 3), g.rperm);
                    return (g.Cf2 && n >= g.nsplit)
                               ? reinterpret_cast<float4*>(g.Cf2 + (size_t)m * g.ldc2 +
                                                           (n - g.nsplit))
                               : reinterpret_cast<float4*>(g.Cf + (size_t)m * g.ldc + n + zoff);
                };
                float4 old[8];
                if (g.accumulate) {
#pragma unroll
                    for (int it = 0; it < 8; ++it) {
                        const int m = m0 + sg::row_pixel(warp * 32 + it * 4 + (lane >> 3), g.rperm);
                        old[it] = m < g.M ? *dst_of(it) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
#pragma unroll
                for (int it = 0; it < 8; ++it) {
                    const int r = it * 4 + (lane >> 3);
                    const int m = m0 + sg::row_pixel(warp * 32 + r, g.rperm);
                    if (m >= g.M) continue;
                    float4 x = *reinterpret_cast<const float4*>(ep + r * 36 + cc);
                    x.x += bn[0];
                    x.y += bn[1];
                    x.z += bn[2];
                    x.w += bn[3];
                    if (g.relu) {
                        x.x = fmaxf(x.x, 0.1f * x.x);
                        x.y = fmaxf(x.y, 0.1f * x.y);
                        x.z = fmaxf(x.z, 0.1f * x.z);
                        x.w = fmaxf(x.w, 0.1f * x.w);
                    }
                    if (g.accumulate) {
                        x.x += old[it].x;
                        x.y += old[it].y;
                        x.z += old[it].z;
                        x.w += old[it].w;
                    }
                    *dst_of(it) = x;
                }
            }
        } else {
            const int n = n0 + c0 + lane;
            const bool col_ok = lane < w && n < g.N;
            const float bn = (col_ok && g.bias) ? g.bias[n] : 0.f;
#pragma unroll 4
            for (int r = 0; r < 32; ++r) {
                const int m = m0 + sg::row_pixel(warp * 32 + r, g.rperm);
                if (!col_ok || m >= g.M) continue;
                float x = ep[r * 36 + lane] + bn;
                if (g.relu) x = fmaxf(x, 0.1f * x);
                float* cf = g.Cf;
                size_t o = (size_t)m * g.ldc + n + zoff;
                if (g.Cf2 && n >= g.nsplit) {
                    cf = g.Cf2;
                    o = (size_t)m * g.ldc2 + (n - g.nsplit);
                }
                if (cf) {
                    if (g.accumulate)
                        cf[o] += x;
                    else
                        cf[o] = x;
                } else {
                    g.Cb[o] = __float2bfloat16_rn(x);
                }
            }
        }
        __syncwarp();
    }
}

// GA: A is the gathered convolution operand (K-major, rows = output pixels); GD: A is the
// gathered data-gradient operand; GAM: A is the gathered convolution operand MN-major (K =
// pixels, M = im2col columns).
// TMA (64 or 32; with GA or GD, both operands K-major): thread 0 alone feeds the stages with
// tiled tensor copies of TMA elements of K per stage (128- or 64-byte swizzled rows): A as one
// box of TMA channels x the tile's 128 pixels (a block of whole rows, or 128 pixels of one row)
// of the activation (GA; the tap's offset applied to the box origin, x1 or x2 by channel) or of
// the output gradient (GD, the offset negated), out-of-image pixels zero-filled by the copy
// itself; B as a TMA x BN box of the weight matrix. Stage s completes on full[s] (transaction
// bytes), is released by the MMAs' commit to empty[s], and STAGES slices are in flight.
// TMA = 1 (with GAM, both operands MN-major): the same feeding for the weight gradient, 64
// pixels of K per stage in 64-byte-swizzled MN-major blocks of 32: A as four boxes of 32
// channels x the 64 pixels (a block of whole rows or 64 pixels of one row), each at its tap's
// offset; B as BN / 32 boxes of 32 output-gradient channels x the same pixels.
template <int BN, int STAGES, bool AMN = false, bool BMN = false, bool GA = false, bool GD = false,
          bool GAM = false, int TMA = 0>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_gemm_tc(const sg::GemmArgs g, int* err, const __grid_constant__ CUtensorMap tmA1,
              const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB) {
    static_assert(!TMA || ((GA || GD) && !AMN && !BMN && (TMA == 64 || TMA == 32)) ||
                      (GAM && AMN && BMN && TMA == 1 && BN % 32 == 0),
                  "TMA feeds the K-major gathers (64 or 32) or the weight gradient (1)");
    constexpr int KS = slice_k(TMA);
    using S = TcShape<BN, STAGES, BMN, KS>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    // 1 KB-aligned base of the stages (the swizzle pattern follows shared-memory address bits)
    const uint32_t raw = su32(smem_raw);
    uint8_t* base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + STAGES * S::STAGE_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int kb = g.kchunk ? blockIdx.z * g.kchunk : 0;
    const int ke = g.kchunk ? min(g.K, kb + g.kchunk) : g.K;
    const int nk = ke > kb ? (ke - kb + KS - 1) / KS : 0;

    sg::pdl_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(tmem_slot)),
                     "r"(tmem_cols(BN))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s <= 2 * STAGES; ++s) mbar_init(su32(bars + s), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_ok = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    sg::pdl_next();
    const uint32_t tmem = *tmem_slot;
    constexpr uint32_t IDESC = idesc_bf16(BM, BN, AMN ? 1 : 0, BMN ? 1 : 0);

    auto stage_a = [&](int s) { return base + s * S::STAGE_BYTES; };
    auto stage_b = [&](int s) { return base + s * S::STAGE_BYTES + S::A_BYTES; };
    // GA / GD: pixel coordinates of the thread's eight A rows, fixed for all K-slices (rows are
    // output pixels, or source pixels at the source's resolution)
    int yx[8], nn[8];
    if (GA || GD) {
        const int RH = GA ? g.conv.H : g.dg.H >> g.dg.up1, RWd = GA ? g.conv.W : g.dg.W >> g.dg.up1;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int p = m0 + (tid >> 3) + 16 * j;
            const int x = p % RWd, q = p / RWd, y = q % RH;
            yx[j] = y | (x << 16);
            nn[j] = p < g.M ? q / RH : -1;
        }
    }
    // GAM: tap and channel of the thread's A column chunk
    int tcol = -1;
    if (GAM) {
        const int col = m0 + 8 * (tid & 15);
        if (col < g.M) {
            const int tap = col >> g.conv.lc;
            tcol = (col & ((1 << g.conv.lc) - 1)) | (tap << 16);
        }
    }
    auto load = [&](int s, int k0) {
        if (GAM)
            load_slice_mn_conv_a(stage_a(s), g.conv, tcol, k0, ke);
        else if (GA)
            load_slice_conv(stage_a(s), g.conv, yx, nn, k0, ke);
        else if (GD)
            load_slice_dgrad(stage_a(s), g.dg, yx, nn, k0, ke);
        else if (AMN)
            load_slice_mn<BM>(stage_a(s), g.A, g.lda, m0, g.M, k0, ke);
        else
            load_slice<BM>(stage_a(s), g.A, g.lda, m0, g.M, k0, ke);
        if (BMN)
            load_slice_mn<BN>(stage_b(s), g.B, g.ldb, n0, g.N, k0, ke);
        else
            load_slice<BN>(stage_b(s), g.B, g.ldb, n0, g.N, k0, ke, g.kperiod);
    };

    bool ok = true;
    if constexpr (TMA) {
        // tile origin: n, y0, x0 of the first of the 128 pixels (a tbh x tbw block); the data
        // gradient of an upsampling convolution has its rows at the source's half resolution
        const int TH = GA || GAM ? g.conv.H : g.dg.H >> g.dg.up1;
        const int TW = GA || GAM ? g.conv.W : g.dg.W >> g.dg.up1;
        const int img = m0 / (TH * TW), rem = m0 - img * (TH * TW);
        const int y0 = rem / TW, x0 = rem - (rem / TW) * TW;
        const int lk = GA || GAM ? g.conv.lc : g.dg.lco;
        auto issue = [&](int st, int k0) {
            const uint32_t full = su32(bars + st);
            if constexpr (GAM) {
                // K = pixels k0 .. k0 + 63: image, row and column of the first
                mbar_expect_tx(full, (uint32_t)(BM * 64 * 2 + BN * 64 * 2));
                const int pn = k0 / (TH * TW), pr = k0 - pn * (TH * TW);
                const int py = pr / TW, px = pr - (pr / TW) * TW;
                if (g.conv.up1) {
                    // upsampling convolution: the slice's 64 pixels (one row segment) in the
                    // order even columns, odd columns (K is summed over, the same order for A
                    // and B); each half reads a run of 32 consecutive source pixels and every
                    // second output-gradient pixel
#pragma unroll
                    for (int b = 0; b < BM / 32; ++b) {
                        const int col = m0 + 32 * b, tap = col >> lk, ci = col & ((1 << lk) - 1);
                        const int dy = tap / 3 - 1, dx = tap - (tap / 3) * 3 - 1;
                        const int sy = (py + dy) >= 0 ? (py + dy) >> 1 : -1;
                        const uint32_t dst = su32(stage_a(st)) + 4096 * b;
                        tma_load_4d(dst, &tmA1, full, ci, (px >> 1) + (dx < 0 ? -1 : 0), sy, pn);
                        tma_load_4d(dst + 2048, &tmA1, full, ci, (px >> 1) + (dx > 0 ? 1 : 0), sy,
                                    pn);
                    }
#pragma unroll
                    for (int b = 0; b < BN / 32; ++b) {
                        const uint32_t dst = su32(stage_b(st)) + 4096 * b;
                        tma_load_4d(dst, &tmB, full, n0 + 32 * b, px, py, pn);
                        tma_load_4d(dst + 2048, &tmB, full, n0 + 32 * b, px + 1, py, pn);
                    }
                    return;
                }
#pragma unroll
                for (int b = 0; b < BM / 32; ++b) {
                    const int col = m0 + 32 * b, tap = col >> lk, ci = col & ((1 << lk) - 1);
                    const int dy = tap / 3 - 1, dx = tap - (tap / 3) * 3 - 1;
                    if (ci < g.conv.C1)
                        tma_load_4d(su32(stage_a(st)) + 4096 * b, &tmA1, full, ci, px + dx,
                                    py + dy, pn);
                    else
                        tma_load_4d(su32(stage_a(st)) + 4096 * b, &tmA2, full, ci - g.conv.C1,
                                    px + dx, py + dy, pn);
                }
#pragma unroll
                for (int b = 0; b < BN / 32; ++b)
                    tma_load_4d(su32(stage_b(st)) + 4096 * b, &tmB, full, n0 + 32 * b, px, py, pn);
                return;
            }
            mbar_expect_tx(full, (uint32_t)(S::A_BYTES + S::B_BYTES));
            const int tap = k0 >> lk, ch = k0 & ((1 << lk) - 1);
            const int dy = tap / 3 - 1, dx = tap - (tap / 3) * 3 - 1;
            if (GA && g.conv.up1) {
                // upsampling layer: the tile's rows come as runs of even, then odd output
                // columns (rperm = half a tile row); each run reads consecutive source pixels of
                // the half-resolution source row floor((y + dy) / 2)
                const int h = g.rperm, tbh = BM / (2 * h);
                for (int i = 0; i < tbh; ++i) {
                    const int yo = y0 + i + dy, sy = yo >= 0 ? yo >> 1 : -1;
                    const uint32_t row = su32(stage_a(st)) + (uint32_t)(i * 2 * h * KS * 2);
                    tma_load_4d(row, &tmA1, full, ch, (x0 >> 1) + (dx < 0 ? -1 : 0), sy, img);
                    tma_load_4d(row + (uint32_t)(h * KS * 2), &tmA1, full, ch,
                                (x0 >> 1) + (dx > 0 ? 1 : 0), sy, img);
                }
            } else if (GA) {
                if (ch < g.conv.C1)
                    tma_load_4d(su32(stage_a(st)), &tmA1, full, ch, x0 + dx, y0 + dy, img);
                else
                    tma_load_4d(su32(stage_a(st)), &tmA2, full, ch - g.conv.C1, x0 + dx, y0 + dy,
                                img);
            } else if (g.dg.up1) {
                // K = (sub-pixel s, tap, channel): the output gradient at (2 y + sy - dy,
                // 2 x + sx - dx), every second pixel in both directions (a strided box)
                const int sub = tap / 9, t9 = tap - sub * 9;
                const int uy = t9 / 3 - 1, ux = t9 - (t9 / 3) * 3 - 1;
                tma_load_4d(su32(stage_a(st)), &tmA1, full, ch, 2 * x0 + (sub & 1) - ux,
                            2 * y0 + (sub >> 1) - uy, img);
            } else {
                tma_load_4d(su32(stage_a(st)), &tmA1, full, ch, x0 - dx, y0 - dy, img);
            }
            tma_load_2d(su32(stage_b(st)), &tmB, full, g.kperiod ? k0 % g.kperiod : k0, n0);
        };
        if (tid == 0) {
            int issued = 0, done_mma = 0;
            bool good = true;
            for (; issued < STAGES && issued < nk; ++issued) issue(issued, kb + issued * KS);
            for (int kt = 0; kt < nk; ++kt) {
                const int st = kt % STAGES;
                if (!mbar_wait(su32(bars + st), (kt / STAGES) & 1)) {
                    good = false;
                    break;
                }
                tc_fence_after();
                // K = 16 per MMA: 32 bytes along a K-major row, or two 512-byte K-groups of an
                // MN-major 64-byte-swizzled block (blocks 4 KB apart)
                constexpr uint32_t HI = GAM || KS == 32 ? desc_hi(512, SW64) : desc_hi(1024, SW128);
                constexpr uint32_t STEP = (GAM ? 1024 : 32) >> 4, LBO = GAM ? 4096 : 16;
                const uint32_t a0 = desc_lo(su32(stage_a(st)), LBO), b0 = desc_lo(su32(stage_b(st)), LBO);
#pragma unroll
                for (int j = 0; j < KS / 16; ++j)
                    tc_mma(tmem, a0 + STEP * j, HI, b0 + STEP * j, HI, IDESC, (kt > 0 || j > 0) ? 1u : 0u);
                tc_commit(su32(bars + STAGES + st));
                done_mma = kt + 1;
                // refill the stage that slice kt - 1 used once its MMAs have read it
                if (kt >= 1 && issued < nk) {
                    const int sp = (kt - 1) % STAGES;
                    if (!mbar_wait(su32(bars + STAGES + sp), ((kt - 1) / STAGES) & 1)) {
                        good = false;
                        break;
                    }
                    issue(sp, kb + issued * KS);
                    ++issued;
                }
            }
            if (!good) {
                // let the copies still in flight land before the CTA may leave (bounded)
                for (int j = done_mma; j < issued; ++j)
                    mbar_wait(su32(bars + j % STAGES), (j / STAGES) & 1);
            }
            if (nk > 0) {
                tc_commit(su32(bars + 2 * STAGES));
                if (!mbar_wait(su32(bars + 2 * STAGES), 0)) good = false;
            }
            if (!good) s_ok = 0;
        }
        __syncthreads();
        ok = s_ok;
    } else {
#pragma unroll 1
    for (int p = 0; p < STAGES - 1; ++p) {
        if (p < nk) load(p, kb + p * BK);
        sg::cp_async_commit();
    }
#pragma unroll 1
    for (int kt = 0; kt < nk; ++kt) {
        const int s = kt % STAGES;
        sg::cp_async_wait<STAGES - 2>();
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            // K = 16 per MMA: 32 bytes along a K-major swizzle row, two 1 KB K-groups of an
            // MN-major block (blocks 8 KB apart)
            constexpr uint32_t HI = desc_hi(1024, SW128);
            const uint32_t a0 = desc_lo(su32(stage_a(s)), AMN ? 8192 : 16);
            const uint32_t b0 = desc_lo(su32(stage_b(s)), BMN ? 8192 : 16);
#pragma unroll
            for (int j = 0; j < BK / 16; ++j)
                tc_mma(tmem, a0 + (AMN ? 128 : 2) * j, HI, b0 + (BMN ? 128 : 2) * j, HI, IDESC,
                       (kt > 0 || j > 0) ? 1u : 0u);
            tc_commit(su32(bars + s));
        }
        const int nxt = kt + STAGES - 1;
        if (nxt < nk && kt >= 1) {
            // the slice being refilled was read by the MMAs of k-tile kt - 1
            if (tid == 0 && !mbar_wait(su32(bars + (kt - 1) % STAGES), ((kt - 1) / STAGES) & 1))
                s_ok = 0;
            __syncthreads();
            if (!s_ok) {
                ok = false;
                break;
            }
        }
        if (nxt < nk) load(nxt % STAGES, kb + nxt * BK);
        sg::cp_async_commit();
    }
    sg::cp_async_wait<0>();
    // completion of every MMA issued (the last commit tracks all earlier ones)
    if (nk > 0) {
        if (tid == 0) {
            tc_commit(su32(bars + 2 * STAGES));
            if (!mbar_wait(su32(bars + 2 * STAGES), 0)) s_ok = 0;
        }
        __syncthreads();
        ok = ok && s_ok;
    }
    }
    if (!ok) {
        if (tid == 0) atomicExch(err, 1);
    } else {
        tc_fence_after();
        // the staging blocks lie in the now idle stage buffers
        epilogue_tile<BN>(g, tmem, reinterpret_cast<float*>(base) + warp * (32 * 36), warp, lane,
                          m0, n0, nk == 0, g.kchunk ? (size_t)blockIdx.z * g.split_stride : 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                     "r"(tmem_cols(BN))
                     : "memory");
    }
}

__host__ __device__ constexpr uint32_t tmem_pow2(int cols) {
    return cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
}

// Sizes of k_wgrad_rows: slices of RA output-gradient rows of 64 pixels (UP: the two row parities, for
// NP column parities) and the ROWS input rows of 72 pixels around them; an MMA's M blocks are BLK
// window rows.
template <int XB, int YB, int CB, bool UP>
struct WgradShape {
    static constexpr int RA = XB == 32 ? 2 : 4, NP = UP ? 2 : 1, ROWS = UP ? 3 : RA + 2;
    static constexpr int BLK = 128 / XB, WROW = 72 * XB * 2, WIN = BLK * WROW, DROW = 64 * YB * 2;
    static constexpr int A_B = CB * WIN, STAGE = A_B + NP * RA * DROW;
    static constexpr int STAGES = STAGE <= 36864 ? 4 : 3;
    static constexpr int N = RA * YB, T = UP ? 4 : 3;  // accumulators per channel block
    static constexpr uint32_t TX = (uint32_t)(CB * ROWS * WROW + NP * RA * DROW);
    static constexpr uint32_t COLS = tmem_pow2(CB * T * N);
    // accumulators the epilogue sums at a time, through the stages' memory
    static constexpr int D = UP ? T : 1;
    static constexpr int RAW = 1024 + STAGES * STAGE + 8 * (2 * STAGES + 1) + 16;
    static constexpr int CTAS = 512 / (int)COLS < 232448 / (RAW + 2048) ? 512 / (int)COLS
                                                                      : 232448 / (RAW + 2048);
    // no more CTAs per SM than its tensor memory holds
    static constexpr int MIN_BYTES = 233472 / (512 / (int)COLS + 1) + 1;
    static constexpr int SMEM = RAW > MIN_BYTES ? RAW : MIN_BYTES;
    static_assert(CB * T * N <= 512 && ROWS <= BLK, "accumulators must fit");
    static_assert(D * N * 128 * 4 <= STAGES * STAGE, "the epilogue's sums must fit the stages");
};

// Weight gradient of a 3 x 3 convolution from staged rows, for CB blocks of XB (32 or 16) input
// channels and YB output channels per CTA (blockIdx.y: which), blockIdx.x one split-K range:
// dW^T[(tap, ci)][co] = sum over pixels p of x(p + off(tap))[ci] dY(p)[co]. Per slice thread 0 loads
// with TMA the input rows y - 1 .. y + RA of pixels x - 4 .. x + 67 (rows of XB channels, swizzled: the
// MN-major layout with K = pixels) and the dY rows y .. y + RA - 1 of 64 pixels. An MMA's M is the
// window's rows (BLK blocks of XB), its N the dY rows (RA blocks of YB), so one MMA per (block, dx, 16
// pixels) holds every (input row, dY row) pair: those with dy = -1, 0, 1 are the taps, summed over the
// dY rows at the end, the rest is dropped (as is what M blocks past the loaded rows read). An A operand
// of 128 x 16 is read from shared memory in 64 cycles, N columns take N / 2: N = 64 or more hides
// what a single dY row (N = 32, three of four M blocks used) spent on operand reads.
// UP: the input has half the resolution (nearest upsampling). Output pixel (2 i + a, 2 j + b) of tap
// (dy, dx) reads input pixel (i + (a + dy) >> 1, j + (b + dx) >> 1), so the products are formed over
// input pixels for the 2 x 2 parities and the two column offsets each reads, 16 products where the
// nine taps over output pixels are 36, and summed into the taps at the end. The dY pixels of one
// column parity come as every second pixel of a box.
// Bound by the MMAs (about 100 cycles for 128 x 64 x 16). 256 x 256 x 8, input -> output channels, before
// (one dY row per MMA from a staged window, or im2col columns fetched per tap) and here, us:
// 32 -> 32 30 / 22, 64 -> 32 82 / 25, 64 -> 32 upsampling 133 / 31; 128 x 128 x 8: 64 -> 64 30 / 24,
// 128 -> 64 60 / 38, 128 -> 64 upsampling 57 / 30. Relative error against FP64 sums of the same operands
// 6.4e-6 / 0.9e-6 at worst (shorter FP32 chains per split).
template <int XB, int YB, int CB, bool UP>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_wgrad_rows(const sg::GemmArgs g, int* err, const __grid_constant__ CUtensorMap tmX1,
                 const __grid_constant__ CUtensorMap tmX2, const __grid_constant__ CUtensorMap tmDY) {
    using S = WgradShape<XB, YB, CB, UP>;
    constexpr int STAGES = S::STAGES, T = S::T, N = S::N, RA = S::RA;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t raw = su32(smem_raw);
    uint8_t* base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + STAGES * S::STAGE);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // kchunk, K: slices
    const int kb = blockIdx.x * g.kchunk, nk = max(0, min(g.K - kb, g.kchunk));
    const int cin = g.conv.C1 + g.conv.C2, ny = g.N / YB;
    const int co0 = (int)(blockIdx.y % ny) * YB, ci0 = (int)(blockIdx.y / ny) * (CB * XB);
    sg::pdl_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(tmem_slot)),
                     "r"(S::COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i <= 2 * STAGES; ++i) mbar_init(su32(bars + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_ok = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    sg::pdl_next();
    const uint32_t tmem = *tmem_slot;
    if (tid == 0) {
        const int segs = (UP ? g.conv.W / 2 : g.conv.W) / 64, rows = g.conv.H / RA;
        auto issue = [&](int st, int k) {
            const uint32_t full = su32(bars + st), a = su32(base + st * S::STAGE);
            mbar_expect_tx(full, S::TX);
            const int r = k / segs, px = (k - r * segs) * 64, n = r / rows, row = r - n * rows;
            const int py = UP ? row : row * RA;
#pragma unroll
            for (int cb = 0; cb < CB; ++cb) {
                const int ci = ci0 + XB * cb;
                if (ci < g.conv.C1)
                    tma_load_4d(a + cb * S::WIN, &tmX1, full, ci, px - 4, py - 1, n);
                else
                    tma_load_4d(a + cb * S::WIN, &tmX2, full, ci - g.conv.C1, px - 4, py - 1, n);
            }
#pragma unroll
            for (int b = 0; b < S::NP; ++b)
                tma_load_4d(a + S::A_B + b * RA * S::DROW, &tmDY, full, co0, UP ? 2 * px + b : px,
                            row * RA, n);
        };
        constexpr uint32_t IDESC = idesc_bf16(BM, N, 1, 1);
        constexpr uint32_t AHI = desc_hi(16 * XB, XB == 32 ? SW64 : SW32);
        constexpr uint32_t BHI = desc_hi(16 * YB, YB == 32 ? SW64 : SW32);
        int issued = 0, done_mma = 0;
        bool good = true;
        for (; issued < STAGES && issued < nk; ++issued) issue(issued, kb + issued);
        for (int kt = 0; kt < nk; ++kt) {
            const int st = kt % STAGES;
            if (!mbar_wait(su32(bars + st), (kt / STAGES) & 1)) {
                good = false;
                break;
            }
            tc_fence_after();
            const uint32_t a = su32(base + st * S::STAGE);
            const uint32_t a0 = desc_lo(a, S::WROW), b0 = desc_lo(a + S::A_B, S::DROW);
#pragma unroll
            for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    // accumulator t: dx = t - 1, or (UP) column parity b and its offset e = 0, 1
                    const int b = UP ? t / 2 : 0, px = UP ? 3 + t / 2 + t % 2 : 3 + t;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        tc_mma(tmem + (uint32_t)((cb * T + t) * N),
                               a0 + (uint32_t)((cb * S::WIN + (px + 16 * j) * XB * 2) >> 4), AHI,
                               b0 + (uint32_t)((b * RA * S::DROW + 16 * j * YB * 2) >> 4), BHI, IDESC,
                               (kt > 0 || j > 0) ? 1u : 0u);
                }
            tc_commit(su32(bars + STAGES + st));
            done_mma = kt + 1;
            if (kt >= 1 && issued < nk) {
                const int sp = (kt - 1) % STAGES;
                if (!mbar_wait(su32(bars + STAGES + sp), ((kt - 1) / STAGES) & 1)) {
                    good = false;
                    break;
                }
                issue(sp, kb + issued);
                ++issued;
            }
        }
        if (!good)
            for (int j = done_mma; j < issued; ++j) mbar_wait(su32(bars + j % STAGES), (j / STAGES) & 1);
        if (nk > 0) {
            tc_commit(su32(bars + 2 * STAGES));
            if (!mbar_wait(su32(bars + 2 * STAGES), 0)) good = false;
        }
        if (!good) s_ok = 0;
    }
    __syncthreads();
    if (!s_ok) {
        if (tid == 0) atomicExch(err, 1);
    } else {
        tc_fence_after();
        const size_t zoff = (size_t)blockIdx.x * g.split_stride;
        float* sum = reinterpret_cast<float*>(base);  // [D][RA][BLK][YB][XB]
        constexpr int CELL = YB * XB;
        const int m = warp * 32 + lane, blk = m / XB, mi = m % XB;
#pragma unroll 1
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll 1
            for (int t0 = 0; t0 < T; t0 += S::D) {
#pragma unroll 1
                for (int c0 = 0; c0 < S::D * N; c0 += 32) {
                    float v[32];
                    if (nk == 0) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = 0.f;
                    } else {
                        tc_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((cb * T + t0) * N + c0), v);
                    }
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int da = (c0 + j) / YB, co = (c0 + j) % YB;  // d RA + a
                        sum[(da * S::BLK + blk) * CELL + co * XB + mi] = v[j];
                    }
                }
                __syncthreads();
                for (int i = tid; i < (UP ? 9 : 3) * CELL; i += TC_THREADS) {
                    const int k = i / CELL, cell = i - k * CELL;
                    const int dyi = UP ? k / 3 : k, dxi = UP ? k - 3 * (k / 3) : t0;
                    float v = 0.f;
                    if (UP) {
#pragma unroll
                        for (int ab = 0; ab < 4; ++ab) {
                            const int a = ab >> 1, b = ab & 1;
                            const int br = 1 + ((a + dyi - 1) >> 1);
                            const int d = 2 * b + ((b + dxi - 1) >> 1) - (b - 1);
                            v += sum[((d * RA + a) * S::BLK + br) * CELL + cell];
                        }
                    } else {
#pragma unroll
                        for (int a = 0; a < RA; ++a) v += sum[(a * S::BLK + dyi + a) * CELL + cell];
                    }
                    const int co = cell / XB, ci = cell - co * XB;
                    g.Cf[(size_t)(co0 + co) * g.ldc + (dyi * 3 + dxi) * cin + ci0 + cb * XB + ci + zoff] = v;
                }
                __syncthreads();
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(S::COLS)
                     : "memory");
    }
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

// 32 bytes to a 32-byte-aligned address: a whole sector per lane
__device__ __forceinline__ void st_global_32B(void* p, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// 32 bytes from a 32-byte-aligned address
__device__ __forceinline__ void ld_global_32B(const void* p, uint32_t (&v)[8]) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                   "=r"(v[7])
                 : "l"(p)
                 : "memory");
}

// a wait for a whole warp: lane 0 polls
__device__ __forceinline__ bool warp_wait(int lane, uint32_t bar, uint32_t parity) {
    int ok = 1;
    if (lane == 0) ok = mbar_wait(bar, parity);
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// Sizes of k_conv_march: rows of 136 pixels of CB blocks of KB channels in a ring, the nine taps'
// weight blocks, mbarriers. UD (GD and UP): a row is its even and its odd columns.
template <int KB, int CB, int BN, bool GD, bool UP>
struct MarchShape {
    static constexpr bool UF = UP && !GD, UD = UP && GD;
    static constexpr int R = UD ? 8 : 6;               // rows in the ring
    static constexpr int G = UF ? 4 : 1;               // tiles (accumulators) per operand row
    static constexpr int ROWB = 136 * KB * 2, SLOT = CB * (UD ? 2 : 1) * ROWB;
    static constexpr int BSUB = BN * KB * 2, WBYTES = 9 * CB * BSUB;
    static constexpr int NBARS = 2 * R + 6;
    static constexpr int SMEM = 1024 + WBYTES + R * SLOT + NBARS * 8;
    // CTAs per SM: two where shared memory allows (232,448 bytes, 1 KB reserved per CTA); registers are
    // fitted to that (the 32 -> 64 data gradient at 256 x 256 x 8 with one CTA of 182 registers 56 us, 38 so)
    static constexpr int PER_SM = 232448 / (SMEM + 2048) >= 2 ? 2 : 1;
};
constexpr int MARCH_THREADS = 192;

// 3 x 3 convolution (GD = false: forward, bias and leaky ReLU, BF16 out) or its data gradient (GD:
// FP32 out, split at nsplit) along a strip 128 operand pixels wide, marching down the rows: every
// operand row is copied to shared memory once (not once per tap and tile), the nine taps' weights
// once per CTA. Each tile of 128 pixels of one row is 9 CB KB / 16 MMAs, whose A operand is a row of
// the ring starting dx pixels aside; the K order is tap, then channel. UP (forward): the operand
// has half the output's resolution (nearest upsampling), and each operand row yields four tiles,
// two output rows of 128 even and 128 odd columns each. UP with GD: a tile is 128 pixels of the
// half-resolution input's gradient, the sum over the 2 x 2 output pixels and nine taps in which each
// takes part (K order: output pixel, tap, channel); four operand rows are read per tile and two
// released, each loaded as its even and its odd columns (every second pixel of a box).
// Roles: warp 4 copies (TMA), warp 5 issues MMAs, warps 0-3 read the finished accumulator (two in
// tensor memory, alternating) and store whole 32-byte sectors, so copies, MMAs and stores of
// neighbouring rows overlap. The data gradient of a source that nothing else reads is not stored in
// FP32 but as that source's finished pre-activation gradient (GemmArgs::rg), whose activation the
// epilogue fetches before it waits for the accumulator, with the bias gradient's sums kept per
// thread until the end: the pass that did this moved 134 MB in 19 us at 256 x 256 x 8, 32 channels.
// Bound by the MMAs' shared-memory reads (a 128 x 16 A slice per
// 16-deep MMA of only BN columns). One 128-pixel tile per CTA with its own window and weights (182 MB
// through L2 for 32 -> 32 channels at 256 x 256 x 8, against 72 MB here) or one box per tap (750 MB for
// 64 -> 32) were bound by that traffic and its latency. 256 x 256 x 8: 32 -> 32 channels 34 -> 23 us, data
// gradient of 64 -> 32 (upsampling) 58 -> 27 (and the leaky-ReLU pass of 12),
// 64 -> 32 (concatenated) 69 -> 44, 64 -> 32 (upsampling) 72 -> 35; 128 x 128 x 8, 64 -> 64: 27 -> 18.
// Waits are polled by one thread each with an iteration limit; a wait that runs out ends its role,
// the others follow by their own limits, copies and MMAs in flight are waited for (bounded).
template <int KB, int CB, int BN, bool GD, bool UP>
__global__ void __launch_bounds__(MARCH_THREADS, MarchShape<KB, CB, BN, GD, UP>::PER_SM)
    k_conv_march(const sg::GemmArgs g, int* err, const __grid_constant__ CUtensorMap tmA1,
                 const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB,
                 int chunk) {
    using S = MarchShape<KB, CB, BN, GD, UP>;
    constexpr bool UF = S::UF, UD = S::UD;
    static_assert((KB == 16 || KB == 32) && BN % 16 == 0 && BN <= 64, "shape");
    constexpr int R = S::R, G = S::G;
    constexpr uint32_t COLS = tmem_pow2(2 * G * BN);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t raw = su32(smem_raw);
    uint8_t* base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    const uint32_t wgt = su32(base), ring = wgt + S::WBYTES, bars = ring + R * S::SLOT;
    auto full = [&](int i) { return bars + 8u * i; };
    auto empty = [&](int i) { return bars + 8u * (R + i); };
    const uint32_t wfull = bars + 8u * (2 * R), done = wfull + 8u;
    auto accf = [&](int b) { return done + 8u + 8u * b; };
    auto acce = [&](int b) { return done + 24u + 8u * b; };
    __shared__ int s_ok;
    __shared__ uint32_t s_tmem;
    __shared__ float s_bias[BN];
    __shared__ float s_col[4][BN];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // the CTA's strip: image, first operand column, operand rows ra .. rb - 1
    const int H = GD ? g.dg.H : g.conv.H, W = GD ? g.dg.W : g.conv.W;
    const int RH = UP ? H / 2 : H, RW = UP ? W / 2 : W;
    const int chunks = (RH + chunk - 1) / chunk, strips = RW / 128;
    const int ck = blockIdx.x % chunks, st = blockIdx.x / chunks;
    const int img = st / strips, x0 = (st - img * strips) * 128;
    const int ra = ck * chunk, rb = min(RH, ra + chunk), n0 = blockIdx.y * BN;

    if (tid == 0) {
        for (int i = 0; i < R; ++i) {
            mbar_init(full(i), 1);
            mbar_init(empty(i), 1);
        }
        mbar_init(wfull, 1);
        mbar_init(done, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf(b), 1);
            mbar_init(acce(b), 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_ok = 1;
    }
    sg::pdl_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(&s_tmem)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (!GD && tid < BN) s_bias[tid] = g.bias ? g.bias[n0 + tid] : 0.f;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    sg::pdl_next();
    const uint32_t tmem = s_tmem;

    if (warp == 4 && lane == 0) {
        // copies: weights, then operand rows ra - 1 .. rb (rows outside the image are zero-filled)
        bool good = true;
        const int rows = (UD ? 2 : 1) * (rb - ra) + 2;
        int issued = 0;
        auto load_row = [&](int i) {
            const int slot = i % R;
            mbar_expect_tx(full(slot), (uint32_t)S::SLOT);
#pragma unroll
            for (int cb = 0; cb < CB; ++cb) {
                const int ci = KB * cb;
                const uint32_t dst = ring + slot * S::SLOT + cb * (UD ? 2 : 1) * S::ROWB;
                if (UD) {  // columns x0 - 4 .. x0 + 67 and x0 + 68 .. x0 + 131 of each parity
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        tma_load_4d(dst + q * S::ROWB, &tmA1, full(slot), ci, 2 * (x0 - 4) + q,
                                    2 * ra - 1 + i, img);
                        tma_load_4d(dst + q * S::ROWB + 72 * KB * 2, &tmA2, full(slot), ci,
                                    2 * (x0 + 68) + q, 2 * ra - 1 + i, img);
                    }
                } else if (GD || ci < g.conv.C1)
                    tma_load_4d(dst, &tmA1, full(slot), ci, x0 - 4, ra - 1 + i, img);
                else
                    tma_load_4d(dst, &tmA2, full(slot), ci - g.conv.C1, x0 - 4, ra - 1 + i, img);
            }
        };
        for (; issued < 3; ++issued) load_row(issued);  // rows >= 3
        mbar_expect_tx(wfull, (uint32_t)S::WBYTES);
        for (int t = 0; t < 9 * CB; ++t) tma_load_2d(wgt + t * S::BSUB, &tmB, wfull, t * KB, n0);
        for (; issued < rows; ++issued) {
            if (issued >= R && !mbar_wait(empty(issued % R), (issued / R - 1) & 1)) {
                good = false;
                break;
            }
            load_row(issued);
        }
        // nothing may still be landing when the CTA leaves
        for (int i = max(0, issued - R); i < issued; ++i) good &= mbar_wait(full(i % R), (i / R) & 1);
        good &= mbar_wait(wfull, 0);
        if (!good) s_ok = 0;
    } else if (warp == 5 && lane == 0) {
        constexpr uint32_t IDESC = idesc_bf16(BM, BN, 0, 0);
        constexpr uint32_t HI = KB == 32 ? desc_hi(512, SW64) : desc_hi(256, SW32);
        const uint32_t w_lo = desc_lo(wgt);
        bool good = mbar_wait(wfull, 0);
        int have = -1;
        for (int r = ra; r < rb && good; ++r) {
            // ring indexes of operand rows r - 1 and r + 1 (UD: 2 r - 1 and 2 r + 2)
            const int it = r - ra, i0 = UD ? 2 * it : it, need = i0 + (UD ? 3 : 2);
            while (have < need && good) {
                ++have;
                good = mbar_wait(full(have % R), (have / R) & 1);
            }
            const int b = it & 1;
            if (good && it >= 2) good = mbar_wait(acce(b), ((it >> 1) - 1) & 1);
            if (!good) break;
            tc_fence_after();
            uint32_t row_lo[UD ? 4 : 3];  // operand rows r - 1, r, r + 1 (UD: 2 r - 1 .. 2 r + 2)
#pragma unroll
            for (int i = 0; i < (UD ? 4 : 3); ++i) row_lo[i] = desc_lo(ring + ((i0 + i) % R) * S::SLOT);
#pragma unroll
            for (int st = 0; st < (UD ? 36 : 9); ++st) {
                const int t = st % 9, sy = st / 18, sx = st / 9 & 1;  // tap and (UD) output pixel
                const int dy = t / 3 - 1, dx = t - (t / 3) * 3 - 1;
#pragma unroll
                for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                    for (int j = 0; j < KB / 16; ++j)
#pragma unroll
                        for (int k = 0; k < G; ++k) {
                            int wr, wc;  // operand row relative to r - 1, column relative to x0 - 4
                            if (UD) {
                                wr = 1 + sy - dy;
                                wc = 4 + ((sx - dx) >> 1) + ((sx - dx) & 1) * 136;  // odd columns follow
                            } else if (UP) {
                                const int yy = (k >> 1) + dy;
                                wr = yy < 0 ? 0 : yy > 1 ? 2 : 1;
                                wc = 4 + ((k & 1) ? (dx > 0 ? 1 : 0) : (dx < 0 ? -1 : 0));
                            } else {
                                wr = 1 + (GD ? -dy : dy);
                                wc = GD ? 4 - dx : 4 + dx;
                            }
                            tc_mma(tmem + (uint32_t)((b * G + k) * BN),
                                   row_lo[wr] + ((wc * KB * 2 + cb * (UD ? 2 : 1) * S::ROWB + 32 * j) >> 4), HI,
                                   w_lo + (((t * CB + cb) * S::BSUB + 32 * j) >> 4), HI, IDESC,
                                   (st > 0 || cb > 0 || j > 0) ? 1u : 0u);
                        }
            }
            tc_commit(accf(b));
            tc_commit(empty(i0 % R));  // operand row r - 1 (UD: 2 r - 1 and 2 r) is not read again
            if (UD) tc_commit(empty((i0 + 1) % R));
        }
        tc_commit(done);
        if (!mbar_wait(done, 0)) good = false;
        if (!good) s_ok = 0;
    } else if (warp < 4) {
        // lane: one pixel of the tile
        const int fuse = GD && g.rg ? min(BN, (g.Cf2 ? g.nsplit : g.N) - n0) : 0;  // columns (may be < 0)
        float acc[GD ? BN : 1] = {};
        uint32_t yv[GD ? BN / 16 : 1][8];
        for (int r = ra; r < rb; ++r) {
            const int b = (r - ra) & 1;
            if (GD) {
                const size_t m = ((size_t)img * RH + r) * RW + x0 + warp * 32 + lane;
#pragma unroll
                for (int c = 0; c < BN; c += 16)
                    if (c < fuse) ld_global_32B(g.ry + m * g.ldc + n0 + c, yv[c / 16]);
            }
            if (!warp_wait(lane, accf(b), ((r - ra) >> 1) & 1)) {
                if (lane == 0) s_ok = 0;
                break;
            }
            tc_fence_after();
            const int px = warp * 32 + lane;
            for (int k = 0; k < G; ++k) {
                const size_t m = UF ? ((size_t)img * H + 2 * r + (k >> 1)) * W + 2 * (x0 + px) + (k & 1)
                                    : ((size_t)img * RH + r) * RW + x0 + px;
#pragma unroll
                for (int c0 = 0; c0 < BN; c0 += 32) {
                    constexpr int CW = BN < 32 ? BN : 32;
                    float v[32];
                    const uint32_t ta =
                        tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((b * G + k) * BN + c0);
                    if (CW == 32)
                        tc_ld32(ta, v);
                    else
                        tc_ld16(ta, v);
                    if (c0 + CW == BN && k == G - 1) {  // the accumulators have been read
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acce(b));
                    }
                    if (!GD) {
#pragma unroll
                        for (int c = 0; c < CW; c += 16) {
                            uint32_t o[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                float a0 = v[c + 2 * i] + s_bias[c0 + c + 2 * i];
                                float a1 = v[c + 2 * i + 1] + s_bias[c0 + c + 2 * i + 1];
                                a0 = fmaxf(a0, 0.1f * a0);
                                a1 = fmaxf(a1, 0.1f * a1);
                                const __nv_bfloat162 h = __floats2bfloat162_rn(a0, a1);
                                o[i] = *reinterpret_cast<const uint32_t*>(&h);
                            }
                            st_global_32B(g.Cb + m * g.ldc + n0 + c0 + c, o);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < CW; c += 16) {
                            if (c0 + c >= fuse) continue;
                            uint32_t o[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const uint32_t yw = yv[(c0 + c) / 16][i];
                                const float2 y =
                                    __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&yw));
                                const float a0 = v[c + 2 * i], a1 = v[c + 2 * i + 1];
                                const __nv_bfloat162 h = __floats2bfloat162_rn(
                                    y.x > 0.f ? a0 : 0.1f * a0, y.y > 0.f ? a1 : 0.1f * a1);
                                const float2 q = __bfloat1622float2(h);
                                acc[c0 + c + 2 * i] += q.x;
                                acc[c0 + c + 2 * i + 1] += q.y;
                                o[i] = *reinterpret_cast<const uint32_t*>(&h);
                            }
                            st_global_32B(g.rg + m * g.ldc + n0 + c0 + c, o);
                        }
#pragma unroll
                        for (int c = 0; c < CW; c += 8) {
                            if (c0 + c < fuse) continue;
                            const int n = n0 + c0 + c;
                            float* dst = g.Cf2 && n >= g.nsplit ? g.Cf2 + m * g.ldc2 + (n - g.nsplit)
                                                                : g.Cf + m * g.ldc + n;
                            uint32_t o[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const float x = g.accumulate ? dst[i] + v[c + i] : v[c + i];
                                o[i] = __float_as_uint(x);
                            }
                            st_global_32B(dst, o);
                        }
                    }
                }
            }
        }
        if (GD && fuse > 0) {
            // the warp's column sums: halves of the columns change places with the lane that sums them
#pragma unroll
            for (int c0 = 0; c0 < BN; c0 += 32) {
                float t[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) t[i] = c0 + i < BN ? acc[(c0 + i) % BN] : 0.f;
#pragma unroll
                for (int h = 16; h > 0; h >>= 1)
#pragma unroll
                    for (int i = 0; i < h; ++i) {
                        const float keep = lane & h ? t[i + h] : t[i], give = lane & h ? t[i] : t[i + h];
                        t[i] = keep + __shfl_xor_sync(0xffffffffu, give, h);
                    }
                if (c0 + lane < BN) s_col[warp][c0 + lane] = t[0];
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && !s_ok) atomicExch(err, 1);
    if (GD && g.rg && tid < BN && n0 + tid < (g.Cf2 ? g.nsplit : g.N))
        g.rpart[(size_t)(n0 + tid) * gridDim.x + blockIdx.x] =
            (s_col[0][tid] + s_col[1][tid]) + (s_col[2][tid] + s_col[3][tid]);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(COLS)
                     : "memory");
    }
}

// The network's first convolution: 8 input channels (16 bytes per pixel), N = 16 or 32 outputs. The
// input window sits in shared memory as it does in memory, one 16-byte row per pixel, which is the
// unswizzled K-major layout: a tap is a start address, and the second eight K of an MMA is the next
// tap, whose distance is the descriptor's lbo. Five MMAs (taps 0+1, 2+3, 4+5, 6+7, 8+zeros) per
// tile of 128 pixels of one row, four rows per CTA from one window of six. Bound by the 64 + 16
// bytes per pixel it moves; gathering 72 columns per pixel with 16-byte copies (k_gemm_tc, two
// 64-wide slices) took 63 us at 256 x 256 x 8 and 32 outputs; this takes 15.
constexpr int C0_ROWS = 4, C0_PITCH = 136;
template <int N>
struct Conv0Shape {
    static constexpr int WIN = (C0_ROWS + 2) * C0_PITCH * 16, ZERO = 128 * 16, WGT = 10 * N * 16;
    // as much as keeps the CTAs of an SM within the 512 tensor-memory columns
    static constexpr int RAW = 128 + WIN + ZERO + WGT;
    static constexpr int MIN_BYTES = 233472 / (512 / (int)tmem_pow2(C0_ROWS * N) + 1) + 1;
    static constexpr int SMEM = RAW > MIN_BYTES ? RAW : MIN_BYTES;
};

template <int N>
__global__ void __launch_bounds__(TC_THREADS)
    k_conv0(const sg::GemmArgs g, int* err, const __grid_constant__ CUtensorMap tmX) {
    using S = Conv0Shape<N>;
    constexpr uint32_t COLS = tmem_pow2(C0_ROWS * N);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t raw = su32(smem_raw);
    uint8_t* base = smem_raw + ((128u - (raw & 127u)) & 127u);
    uint8_t* wgt = base + S::WIN + S::ZERO;
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_ok;
    __shared__ float s_bias[N];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H = g.conv.H, W = g.conv.W, strips = W / 128, bands = H / C0_ROWS;
    const int st = blockIdx.x % strips, q = blockIdx.x / strips, band = q % bands, img = q / bands;
    const int x0 = st * 128, y0 = band * C0_ROWS;
    if (tid == 0) {
        mbar_init(su32(bars), 1);
        mbar_init(su32(bars + 1), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_ok = 1;
    }
    // zeros behind the window: the K = 72 .. 79 half of the last MMA
    for (int i = tid; i < S::ZERO / 16; i += TC_THREADS)
        reinterpret_cast<uint4*>(base + S::WIN)[i] = make_uint4(0, 0, 0, 0);
    sg::pdl_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(&s_tmem)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    // weights [n][tap][8] as core matrices of eight n: tap-major, then n / 8; tap 9 is zero
    for (int i = tid; i < 10 * N; i += TC_THREADS) {
        const int tap = i / N, n = i - tap * N;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (tap < 9) v = *reinterpret_cast<const uint4*>(g.B + (size_t)n * 72 + tap * 8);
        *reinterpret_cast<uint4*>(wgt + i * 16) = v;
    }
    if (tid < N) s_bias[tid] = g.bias[tid];
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    sg::pdl_next();
    const uint32_t tmem = s_tmem;
    if (tid == 0) {
        const uint32_t full = su32(bars), fin = su32(bars + 1), win = su32(base);
        mbar_expect_tx(full, (uint32_t)S::WIN);
        tma_load_4d(win, &tmX, full, 0, x0 - 4, y0 - 1, img);
        bool good = mbar_wait(full, 0);
        if (good) {
            tc_fence_after();
            constexpr uint32_t HI = desc_hi(128, SW_NONE), IDESC = idesc_bf16(BM, N, 0, 0);
            const uint32_t zero = win + S::WIN;
#pragma unroll
            for (int r = 0; r < C0_ROWS; ++r)
#pragma unroll
                for (int p = 0; p < 5; ++p) {
                    const int t = 2 * p, u = 2 * p + 1;
                    const uint32_t a = win + ((r + t / 3) * C0_PITCH + 3 + t % 3) * 16;
                    const uint32_t b = u < 9 ? win + ((r + u / 3) * C0_PITCH + 3 + u % 3) * 16 : zero;
                    tc_mma(tmem + (uint32_t)(r * N), desc_lo(a, b - a), HI,
                           desc_lo(su32(wgt) + t * N * 16, N * 16), HI, IDESC, p > 0 ? 1u : 0u);
                }
            tc_commit(fin);
            good = mbar_wait(fin, 0);
        } else {
            mbar_wait(full, 0);  // let the copy land (bounded)
        }
        if (!good) s_ok = 0;
    }
    __syncthreads();
    if (!s_ok) {
        if (tid == 0) atomicExch(err, 1);
    } else {
        tc_fence_after();
#pragma unroll
        for (int r = 0; r < C0_ROWS; ++r) {
            float v[32];
            const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(r * N);
            if (N == 32)
                tc_ld32(ta, v);
            else
                tc_ld16(ta, v);
            const size_t m = ((size_t)img * H + y0 + r) * W + x0 + warp * 32 + lane;
#pragma unroll
            for (int c = 0; c < N; c += 16) {
                uint32_t o[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float a0 = v[c + 2 * i] + s_bias[c + 2 * i];
                    float a1 = v[c + 2 * i + 1] + s_bias[c + 2 * i + 1];
                    a0 = fmaxf(a0, 0.1f * a0);
                    a1 = fmaxf(a1, 0.1f * a1);
                    const __nv_bfloat162 h = __floats2bfloat162_rn(a0, a1);
                    o[i] = *reinterpret_cast<const uint32_t*>(&h);
                }
                st_global_32B(g.Cb + m * N + c, o);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(COLS)
                     : "memory");
    }
}

// Its weight gradient, dW^T[(tap, ci)][co] = sum over pixels x(p + off(tap))[ci] dY(p)[co], from the
// same 16-byte pixel rows: as an unswizzled MN-major operand the next eight M are the pixel 16
// bytes on, i.e. the next dx, so one MMA of M = 128 covers dx = -1, 0, 1 (blocks 0-2; the other
// blocks read further pixels and their rows are dropped), with one accumulator per dy. Slices of 128
// pixels of one row (K), each CTA one split-K range of them; the partial is stored as
// [co][tap][ci]. 256 x 256 x 8, 32 outputs: 98 us with the 72 columns gathered per pixel, 24 here.
template <int N>
struct Wgrad0Shape {
    static constexpr int STAGES = 4, WIN = 3 * C0_PITCH * 16, DY = 128 * N * 2, STAGE = WIN + DY;
    // window sizes are multiples of 128 bytes, so every dY block stays aligned to its swizzle when
    // the dY blocks come first; 512 bytes behind the last window for the dropped rows' reads
    static constexpr int SMEM = 1024 + STAGES * STAGE + 512 + 8 * (2 * STAGES + 1);
};
template <int N>
__global__ void __launch_bounds__(TC_THREADS)
    k_wgrad0(const sg::GemmArgs g, int* err, const __grid_constant__ CUtensorMap tmX,
             const __grid_constant__ CUtensorMap tmDY) {
    using S = Wgrad0Shape<N>;
    constexpr int STAGES = S::STAGES;
    constexpr uint32_t COLS = tmem_pow2(3 * N);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t raw = su32(smem_raw);
    uint8_t* base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    auto dyb = [&](int st) { return su32(base) + st * S::DY; };
    auto win = [&](int st) { return su32(base) + STAGES * S::DY + st * S::WIN; };
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + STAGES * S::STAGE + 512);
    __shared__ uint32_t s_tmem;
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kb = blockIdx.x * g.kchunk, ke = min(g.K, kb + g.kchunk);
    const int nk = ke > kb ? (ke - kb) / 128 : 0;
    if (tid == 0) {
        for (int i = 0; i <= 2 * STAGES; ++i) mbar_init(su32(bars + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_ok = 1;
    }
    sg::pdl_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(&s_tmem)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    sg::pdl_next();
    const uint32_t tmem = s_tmem;
    const int H = g.conv.H, W = g.conv.W;
    auto issue = [&](int st, int k0) {
        const uint32_t full = su32(bars + st);
        mbar_expect_tx(full, (uint32_t)S::STAGE);
        const int pn = k0 / (H * W), pr = k0 - pn * (H * W), py = pr / W, px = pr - py * W;
        tma_load_4d(win(st), &tmX, full, 0, px - 4, py - 1, pn);
        tma_load_4d(dyb(st), &tmDY, full, 0, px, py, pn);
    };
    if (tid == 0) {
        constexpr uint32_t IDESC = idesc_bf16(BM, N, 1, 1), AHI = desc_hi(16, SW_NONE);
        constexpr uint32_t BHI = N == 32 ? desc_hi(512, SW64) : desc_hi(256, SW32);
        int issued = 0, done_mma = 0;
        bool good = true;
        for (; issued < STAGES && issued < nk; ++issued) issue(issued, kb + issued * 128);
        for (int kt = 0; kt < nk; ++kt) {
            const int st = kt % STAGES;
            if (!mbar_wait(su32(bars + st), (kt / STAGES) & 1)) {
                good = false;
                break;
            }
            tc_fence_after();
            const uint32_t a0 = desc_lo(win(st) + 3 * 16, 128), b0 = desc_lo(dyb(st), 4096);
#pragma unroll
            for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    tc_mma(tmem + (uint32_t)(dy * N), a0 + dy * C0_PITCH + 16 * j, AHI,
                           b0 + (uint32_t)((j * 16 * N * 2) >> 4), BHI, IDESC, (kt > 0 || j > 0) ? 1u : 0u);
            tc_commit(su32(bars + STAGES + st));
            done_mma = kt + 1;
            if (kt >= 1 && issued < nk) {
                const int sp = (kt - 1) % STAGES;
                if (!mbar_wait(su32(bars + STAGES + sp), ((kt - 1) / STAGES) & 1)) {
                    good = false;
                    break;
                }
                issue(sp, kb + issued * 128);
                ++issued;
            }
        }
        if (!good)
            for (int j = done_mma; j < issued; ++j) mbar_wait(su32(bars + j % STAGES), (j / STAGES) & 1);
        if (nk > 0) {
            tc_commit(su32(bars + 2 * STAGES));
            if (!mbar_wait(su32(bars + 2 * STAGES), 0)) good = false;
        }
        if (!good) s_ok = 0;
    }
    __syncthreads();
    if (!s_ok) {
        if (tid == 0) atomicExch(err, 1);
    } else if (warp == 0) {
        // lane: block dx = lane / 8 - 1 (the first three), channel lane % 8
        tc_fence_after();
        float* out = g.Cf + (size_t)blockIdx.x * g.split_stride;
#pragma unroll 1
        for (int dy = 0; dy < 3; ++dy) {
            float v[32];
            if (nk == 0) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = 0.f;
            } else if (N == 32) {
                tc_ld32(tmem + (uint32_t)(dy * N), v);
            } else {
                tc_ld16(tmem + (uint32_t)(dy * N), v);
            }
            if (lane < 24)
#pragma unroll
                for (int n = 0; n < N; ++n) out[n * 72 + dy * 24 + lane] = v[n];
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(COLS)
                     : "memory");
    }
}

}  // namespace sgtc
}  // namespace lbm

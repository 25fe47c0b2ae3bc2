// Deterministic sums over lattice fields, shared by the reductions and the batched residual.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbm {

// Exact sums of FP32 values in [2^-13, 2^9) with 32-bit integers: such a value v is a whole number
// of 2^-36, and v = hi 2^-13 + lo 2^-36 with whole |hi| <= 2^22 and |lo| <= 2^22, both read off
// the bits of an FP32 sum with a suitable power of two (whose last bit is worth 2^-13, 2^-36).
// That is six operations of the FP32 and integer pipes per value, where the FP64 pipe of this chip
// takes two lanes per cycle and SM. Everything else (zero, negative, tiny, huge, not finite) is
// left to FP64.
constexpr unsigned kFixLo = 0x39000000u, kFixRange = 0x44000000u - 0x39000000u;  // 2^-13, 2^9
__device__ __forceinline__ unsigned fix_key(float v) { return __float_as_uint(v) - kFixLo; }
__device__ __forceinline__ bool fix_ok(float v) { return fix_key(v) < kFixRange; }
struct Fix {
    int hi, lo;
};
__device__ __forceinline__ Fix to_fix(float v) {
    const float mh = 1536.f, ml = 1.5f / 8192.f;  // 1.5 * 2^10 and 1.5 * 2^-13
    const float h = __fadd_rn(v, mh);
    const float rest = __fsub_rn(v, __fsub_rn(h, mh));  // exact
    const float l = __fadd_rn(rest, ml);                // exact
    return Fix{__float_as_int(h) - __float_as_int(mh), __float_as_int(l) - __float_as_int(ml)};
}
constexpr double kFixUnit = 1.0 / 68719476736.0;  // 2^-36
// values a thread may add to its 32-bit halves before they move on (255 * 2^22 < 2^30)
constexpr int kFixMost = 255;

// Sum of one thread: exact part in units of 2^-36 (running 32-bit halves and their 64-bit total) and FP64
// part. A total passes to the FP64 part once it exceeds 2^52, and at most 255 values of less than 2^45
// are added between two looks at it, so it stays below 2^54 and the sum over a block of up to 256
// threads below 2^62. Exact within a block as long as no thread's total has passed on.
struct FixSum {
    int hi = 0, lo = 0, n = 0;
    long long fix = 0;
    double acc = 0;
    __device__ __forceinline__ void settle() {
        fix += (long long)hi * (1 << 23) + lo;
        hi = lo = 0;
    }
    __device__ __forceinline__ void make_room(int more) {
        n += more;
        if ((n & ~kFixMost) != 0) {
            settle();
            n = more;
            if (fix > (1ll << 52)) {
                acc += (double)fix * kFixUnit;
                fix = 0;
            }
        }
    }
    __device__ __forceinline__ void add(const Fix& f) {
        hi += f.hi;
        lo += f.lo;
    }
};

__device__ __forceinline__ void load4(const float* g, float* v) {
    const float4 a = *reinterpret_cast<const float4*>(g);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void load4(const double* g, double* v) {
    const double2 a = *reinterpret_cast<const double2*>(g);
    const double2 b = *(reinterpret_cast<const double2*>(g) + 1);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
template <typename T>
__device__ __forceinline__ void load8(const T* g, T* v) {
    load4(g, v);
    load4(g + 4, v + 4);
}

template <typename V>
__device__ __forceinline__ V warp_sum(V v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Total of the threads' FixSums over a block of up to 256 threads in a fixed order, valid in thread
// 0 (two barriers; the FP64 halves are only added where some thread has one).
__device__ __forceinline__ double block_sum(FixSum& v, long long* s_fix, double* s_acc) {
    v.settle();
    const int warps = blockDim.x >> 5;
    const int has_acc = __syncthreads_or(v.acc != 0.0);  // true for NaN
    const long long f = warp_sum(v.fix);
    if ((threadIdx.x & 31) == 0) s_fix[threadIdx.x >> 5] = f;
    if (has_acc) {
        const double a = warp_sum(v.acc);
        if ((threadIdx.x & 31) == 0) s_acc[threadIdx.x >> 5] = a;
    }
    __syncthreads();
    if (threadIdx.x != 0) return 0.0;
    long long ft = 0;
    for (int w = 0; w < warps; ++w) ft += s_fix[w];
    double t = (double)ft * kFixUnit;
    if (has_acc)
        for (int w = 0; w < warps; ++w) t += s_acc[w];
    return t;
}

// True in every thread of the block that is the last of `blocks` to get here; what the others
// wrote before is then visible to it. Resets the ticket for the next launch.
__device__ __forceinline__ bool last_block(unsigned* ticket, unsigned blocks, int* s_last) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        *s_last = atomicAdd(ticket, 1u) == blocks - 1;
        if (*s_last) *ticket = 0;
    }
    __syncthreads();
    if (*s_last) __threadfence();
    return *s_last != 0;
}

}  // namespace lbm

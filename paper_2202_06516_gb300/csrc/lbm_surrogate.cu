// Learned warm start: a convolutional U-Net that maps (solid mask, wall-wetting map, drop-volume
// plane) on an H x W lattice to a near-equilibrium density field, trained on equilibrated fields
// the solver generates. The paper has no such component; it shortens the plain relaxation from a
// flat-cap start (Sec. 4, Eq. 16) that the solver otherwise performs.
//
// Network (levels l = 1..4, channels c_l = base * 2^(l-1)):
//   encoder   conv3x3 + leaky ReLU (slope 0.1) twice per level, 2x2 average pooling between
//   decoder   2x upsampling folded into the next conv3x3 (nearest), the skip concatenation folded
//             into the following conv3x3 (two-source im2col), conv3x3 + leaky ReLU twice per level
//   head      1x1 conv to one channel, sigmoid: phi = (rho - rho_g) / (rho_l - rho_g)
// Activations BF16 NHWC, weights FP32 masters with BF16 copies, all contractions on the tcgen05
// tensor cores with FP32 accumulation in tensor memory (sg_tc.cuh), as implicit GEMMs whose
// operands are the 3 x 3 neighbourhoods of the activations: the forward convolution, the
// weight gradient (pixels as K; an im2col buffer only when the resolution is not a power of two
// and the rows do not suit k_wgrad_rows) and the data gradient (output gradients around each source
// pixel). Where the shapes allow, the operands arrive as tensor-map (TMA) boxes built once per
// network (make_tensor_maps). Levels of 16 to 64 channels with rows of 128 pixels march down a ring of
// staged rows (k_conv_march), their weight gradients take rows of 64 pixels (k_wgrad_rows), the first
// convolution reads the input once (k_conv0, k_wgrad0). Other layers fetch a box per tap (k_gemm_tc:
// the tap's offset moves the box, the image border is zero-filled, upsampling layers order their
// rows or K even/odd or read every second pixel), or their loaders gather with cp.async.
// Loss: masked mean squared error on phi. Optimiser: Adam.
#include <math.h>

#include <algorithm>
#include <string>
#include <vector>

#include "lbm_internal.cuh"
#include "lbm_trace.h"
#include "sg_gemm.cuh"
#include "sg_tc.cuh"

#include <atomic>
#include <mutex>

namespace lbm {
void set_global_error(const std::string& msg);
}

using bf16 = __nv_bfloat16;

namespace lbm {
namespace sg {
namespace {

constexpr int kT = 256;
constexpr int kReluBlocks = 1024;  // blocks of the fused leaky-ReLU adjoint / bias-sum pass

int blocks_for(long long n) {
    long long b = (n + kT - 1) / kT;
    return (int)(b > 65535LL * 8 ? 65535LL * 8 : (b < 1 ? 1 : b));
}

// Pixel index p -> (n, y, x) of a batch of H x W images (NHWC); P2: H and W are powers of two
// and the split is done with shifts and masks.
struct PixDims {
    int H, W, lh, lw;  // lh, lw: log2 H, log2 W when P2
};

template <bool P2>
__device__ __forceinline__ void pix_split(int p, const PixDims& d, int& n, int& y, int& x) {
    if (P2) {
        x = p & (d.W - 1);
        y = (p >> d.lw) & (d.H - 1);
        n = p >> (d.lw + d.lh);
    } else {
        x = p % d.W;
        const int q = p / d.W;
        y = q % d.H;
        n = q / d.H;
    }
}

// im2col of a 3x3, pad-1 convolution whose input channels are [source 1 | source 2]:
// col[p][(ky*3+kx)*C + c] = x(n, y+ky-1, x+kx-1, c). Source 1 may be stored at half resolution
// (up1 = 1: nearest 2x upsampling on the fly). Eight channels per thread (16-byte accesses); the
// number of 8-channel groups C / 8 = 2^lc8, so thread t writes the 16 bytes at col + 8 t.
template <bool P2>
__global__ void k_im2col(const bf16* x1, int C1, int up1, const bf16* x2, int C2, PixDims d,
                         int P, int lc8, bf16* col) {
    pdl_next();
    pdl_wait();
    const int C8 = 1 << lc8;
    const long long total = (long long)P * 9 * C8;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int c8 = (int)(t & (C8 - 1));
        const int tq = (int)(t >> lc8);  // p * 9 + tap
        const int p = tq / 9, tap = tq - p * 9;
        int n, yy, xx;
        pix_split<P2>(p, d, n, yy, xx);
        const int sy = yy + tap / 3 - 1, sx = xx + tap % 3 - 1;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (sy >= 0 && sy < d.H && sx >= 0 && sx < d.W) {
            const int c = c8 * 8;
            if (c < C1) {
                const int h1 = up1 ? d.H / 2 : d.H, w1 = up1 ? d.W / 2 : d.W;
                const int ty = up1 ? sy >> 1 : sy, tx = up1 ? sx >> 1 : sx;
                v = *reinterpret_cast<const uint4*>(x1 + (((size_t)n * h1 + ty) * w1 + tx) * C1 + c);
            } else {
                v = *reinterpret_cast<const uint4*>(x2 + (((size_t)n * d.H + sy) * d.W + sx) * C2 +
                                                    (c - C1));
            }
        }
        *reinterpret_cast<uint4*>(col + (size_t)t * 8) = v;
    }
}

// 2 x 2 average pool, eight channels per thread (16-byte accesses; C / 8 = 2^lc8). Bound by its 10
// bytes per output element of traffic; one channel per thread with 64-bit index divisions took 36 us
// on the 32-channel 256 x 256 x 8 map (42 MB).
__global__ void __launch_bounds__(kT)
    k_avgpool(const bf16* x, bf16* y, long long n8, int H, int W, int lc8) {
    pdl_next();
    pdl_wait();
    const int h = H / 2, w = W / 2, C = 8 << lc8;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n8;
         t += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(t & ((1 << lc8) - 1)) * 8;
        const int q = (int)(t >> lc8), X = q % w, r = q / w, Y = r % h, n = r / h;
        const bf16* src = x + (((size_t)n * H + 2 * Y) * W + 2 * X) * C + c;
        const uint4 v[4] = {*reinterpret_cast<const uint4*>(src),
                            *reinterpret_cast<const uint4*>(src + C),
                            *reinterpret_cast<const uint4*>(src + (size_t)W * C),
                            *reinterpret_cast<const uint4*>(src + (size_t)W * C + C)};
        uint4 out;
        __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(&out);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 f = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&v[k])[i]);
                s.x = k ? s.x + f.x : f.x;
                s.y = k ? s.y + f.y : f.y;
            }
            o[i] = __floats2bfloat162_rn(0.25f * s.x, 0.25f * s.y);
        }
        reinterpret_cast<uint4*>(y)[t] = out;
    }
}

// Number of non-zero bytes of the loss mask, added to *cnt (integer atomics: exact)
__global__ void __launch_bounds__(kT) k_mask_count(const uint8_t* mask, long long n, int* cnt) {
    pdl_next();
    pdl_wait();
    int c = 0;
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n16 = ((uintptr_t)mask & 15) == 0 ? n / 16 : 0;
    for (long long t = t0; t < n16; t += stride) {
        const uint4 v = reinterpret_cast<const uint4*>(mask)[t];
        c += __popc(__vcmpne4(v.x, 0u)) + __popc(__vcmpne4(v.y, 0u)) + __popc(__vcmpne4(v.z, 0u)) +
             __popc(__vcmpne4(v.w, 0u));
    }
    c /= 8;
    for (long long t = 16 * n16 + t0; t < n; t += stride) c += mask[t] != 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(cnt, c);
}

// The leaky-ReLU adjoint of one convolution's output fused with what feeds it and what reads
// it: g = (dy + dyp / 4) * (y > 0 ? 1 : 0.1), stored as BF16 for the gradient GEMMs, where dyp
// (POOL) is the gradient of the 2 x 2 average pool taken of this output, whose adjoint gives a
// quarter to each of the four source pixels (added after the other consumers' contributions,
// as a separate pass would); and the per-block column sums of the stored g (the bias gradient's
// partials). MODE 2: dy is the head's, the product of the pixel's dz and the head weight hw[c], formed
// here instead of being written and read as a tensor. Thread t always covers the eight channels 8 t mod C (8 x threads per block is a
// multiple of C), so each block adds its threads' sums per channel in thread order into
// part[c][block] (deterministic). H, W: the output resolution (even when POOL).
// MODE 0: dy alone, 1: with the pool's gradient (POOL), 2: dy[p] hw[c].
template <int MODE>
__global__ void k_relu_bias(const float* dy, const float* dyp, const float* hw, const bf16* y,
                            bf16* g, long long n8, int C, int H, int W, float* part) {
    pdl_next();
    pdl_wait();
    constexpr bool POOL = MODE == 1;
    __shared__ float sred[kT * 8];
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n8;
         t += (long long)gridDim.x * blockDim.x) {
        const uint4 yv = reinterpret_cast<const uint4*>(y)[t];
        float d[8];
        if (MODE == 2) {
            const long long e = 8 * t, p = e / C;
            const int c = (int)(e - p * C);
            const float dz = dy[p];
#pragma unroll
            for (int j = 0; j < 8; ++j) d[j] = dz * hw[c + j];
        } else {
            const float4 a = reinterpret_cast<const float4*>(dy)[2 * t];
            const float4 b = reinterpret_cast<const float4*>(dy)[2 * t + 1];
            d[0] = a.x, d[1] = a.y, d[2] = a.z, d[3] = a.w;
            d[4] = b.x, d[5] = b.y, d[6] = b.z, d[7] = b.w;
        }
        if (POOL) {
            const long long e = 8 * t, p = e / C;
            const int c = (int)(e - p * C);
            const long long q = p / W, n = q / H;
            const int xx = (int)(p - q * W), yy = (int)(q - n * H);
            const float4* src = reinterpret_cast<const float4*>(
                dyp + (((n * (H / 2) + yy / 2) * (W / 2) + xx / 2) * C + c));
            const float4 pa = src[0], pb = src[1];
            const float pv[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) d[j] += 0.25f * pv[j];
        }
        const __nv_bfloat162* yh = reinterpret_cast<const __nv_bfloat162*>(&yv);
        uint4 out;
        __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&out);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 yf = __bfloat1622float2(yh[i]);
            const float g0 = yf.x > 0.f ? d[2 * i] : 0.1f * d[2 * i];
            const float g1 = yf.y > 0.f ? d[2 * i + 1] : 0.1f * d[2 * i + 1];
            oh[i] = __floats2bfloat162_rn(g0, g1);
            const float2 r = __bfloat1622float2(oh[i]);
            acc[2 * i] += r.x;
            acc[2 * i + 1] += r.y;
        }
        reinterpret_cast<uint4*>(g)[t] = out;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) sred[threadIdx.x * 8 + j] = acc[j];
    __syncthreads();
    // channel c: the threads c / 8 + k C / 8 (k = 0, 1, ...), slot c % 8
    const int groups = C / 8, reps = blockDim.x / groups;
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        float s = 0.f;
        for (int k = 0; k < reps; ++k) s += sred[(c / 8 + k * groups) * 8 + (c & 7)];
        part[(size_t)c * gridDim.x + blockIdx.x] = s;
    }
}

// out[c] = sum over b of the partials of column c: part[b * C + c], or part[c * nb + b] when
// transposed; one block per column, a fixed-shape tree in shared memory (deterministic). loss (the
// head's sums: weights, loss, bias): the last but one column goes to *loss and the last takes its
// place in out.
__global__ void k_colsum_final(const float* part, int nb, int C, float* out, int transposed,
                               float* loss) {
    pdl_next();
    pdl_wait();
    __shared__ float sm[kT];
    const int c = blockIdx.x;
    float s = 0.f;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        s += transposed ? part[(size_t)c * nb + b] : part[(size_t)b * C + c];
    sm[threadIdx.x] = s;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) sm[threadIdx.x] += sm[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    if (loss && c == C - 2)
        *loss = sm[0];
    else
        out[loss && c == C - 1 ? c - 1 : c] = sm[0];
}

// head: phi = sigmoid(sum_c x[p][c] w[c] + b); with targets, also the loss terms and the
// gradient: dz = 2 m (phi - t) phi (1 - phi) / n_mask (the input's gradient is dz w[c], formed by
// the pass that reads it); per-block partial sums of loss, dz * x[p][c] (weight gradient) and dz
// (bias gradient) for a deterministic reduction. n_mask: the device's count of loss pixels.
template <int C>
__global__ void k_head(const bf16* x, const float* w, const float* bptr, float* phi, long long P,
                       const float* target, const uint8_t* mask, const int* n_mask, float* dzp,
                       float* part /* per block: C + 2 */) {
    pdl_next();
    pdl_wait();
    __shared__ float sw[C];
    __shared__ float red[kT / 32][C + 2];
    for (int c = threadIdx.x; c < C; c += blockDim.x) sw[c] = w[c];
    __syncthreads();
    const float b = *bptr;
    const int cnt = target ? *n_mask : 0;
    const float inv_n = cnt > 0 ? 1.f / (float)cnt : 0.f;
    float acc[C + 2];
#pragma unroll
    for (int c = 0; c < C + 2; ++c) acc[c] = 0.f;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P;
         p += (long long)gridDim.x * blockDim.x) {
        float z = b;
        float xv[C];
        // the pixel's C channels as 16-byte vectors (C is a multiple of 8)
#pragma unroll
        for (int v = 0; v < C / 8; ++v) {
            const uint4 raw = reinterpret_cast<const uint4*>(x + p * C)[v];
            const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f2 = __bfloat1622float2(h[i]);
                xv[8 * v + 2 * i] = f2.x;
                xv[8 * v + 2 * i + 1] = f2.y;
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) z += xv[c] * sw[c];
        const float f = 1.f / (1.f + __expf(-z));
        phi[p] = f;
        if (target) {
            const float m = mask[p] ? 1.f : 0.f;
            const float e = f - target[p];
            const float dz = 2.f * m * e * f * (1.f - f) * inv_n;
            acc[C] += m * e * e * inv_n;
            acc[C + 1] += dz;
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] += dz * xv[c];
            dzp[p] = dz;
        }
    }
    if (!target) return;
#pragma unroll
    for (int c = 0; c < C + 2; ++c) {
        float v = acc[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][c] = v;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < C + 2; c += blockDim.x) {
        float s = 0.f;
        for (int q = 0; q < kT / 32; ++q) s += red[q][c];
        part[(size_t)blockIdx.x * (C + 2) + c] = s;
    }
}

// Offsets and shapes of the convolution weights in the parameter vector, for the kernels that
// keep the BF16 copies (the forward/weight-gradient layout w[co][tap][ci] and the data-gradient
// layout wd[ci][tap][co]).
struct ConvTable {
    int n;
    long long off[24];
    int cout[24], cin[24];
    int tile[25];  // first block of each convolution in k_adam
};
// Bias gradients to finish: per convolution the partial sums part[c * nb + b], its first column
// among all of them and where its sums go.
struct BiasTable {
    int n;
    int col[25], nb[24];
    const float* part[24];
    float* out[24];
};

// BF16 copies of parameter t with FP32 value x: wb[t], and for a convolution weight also its
// data-gradient position wd[off + (ci 9 + tap) cout + co]
__device__ __forceinline__ void store_bf16_copies(long long t, float x, bf16* wb, bf16* wd,
                                                  const ConvTable& tab) {
    const bf16 h = __float2bfloat16_rn(x);
    wb[t] = h;
    for (int k = 0; k < tab.n; ++k) {
        const long long loc = t - tab.off[k];
        const long long len = (long long)tab.cout[k] * 9 * tab.cin[k];
        if (loc >= 0 && loc < len) {
            const int cin = tab.cin[k], cout = tab.cout[k];
            const int co = (int)(loc / (9 * cin)), rem = (int)(loc - (long long)co * 9 * cin);
            const int tap = rem / cin, ci = rem - tap * cin;
            wd[tab.off[k] + ((long long)ci * 9 + tap) * cout + co] = h;
            return;
        }
    }
}

// The bias gradients of all listed convolutions in one launch, one warp per column (each alone was a
// launch of 5.6 us on one block per column). Bound by reading the partials, 4 KB per column.
__global__ void k_bias_final(const BiasTable tab) {
    pdl_next();
    pdl_wait();
    const int col = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
    if (col >= tab.col[tab.n]) return;
    int k = 0;
    while (col >= tab.col[k + 1]) ++k;
    const int c = col - tab.col[k], nb = tab.nb[k];
    const float* p = tab.part[k] + (size_t)c * nb;
    float s = 0.f;
#pragma unroll 8
    for (int b = lane; b < nb; b += 32) s += p[b];
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) s += __shfl_xor_sync(0xffffffffu, s, h);
    if (lane == 0) tab.out[k][c] = s;
}

// Adam with bias correction (c1, c2 = 1 / (1 - beta^t)) and the BF16 copies of the updated
// parameters. A block takes 32 outputs x 32 inputs (tap, ci) of one convolution and passes the BF16
// weights through shared memory, so that both copies are written along their rows: writing the
// data-gradient copy element by element (2 bytes every 18 C_in) took 33 us for 2.1 M parameters,
// 15 here. The blocks of a convolution's first inputs also take its biases, block 0 the head.
__global__ void __launch_bounds__(256)
    k_adam(float* w, const float* g, float* m, float* v, long long n, int nhead, float lr, float b1,
           float b2, float eps, float c1, float c2, bf16* wb, bf16* wd, const ConvTable tab) {
    pdl_next();
    __shared__ bf16 sm[32][34];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int k = 0;
    while ((int)blockIdx.x >= tab.tile[k + 1]) ++k;
    const int cin = tab.cin[k], cout = tab.cout[k], K = 9 * cin, kt = (K + 31) / 32;
    const int tile = blockIdx.x - tab.tile[k], co0 = tile / kt * 32, k0 = tile % kt * 32;
    pdl_wait();
    auto step = [&](long long t, float gi, float mo, float vo, float wo) {
        const float mi = b1 * mo + (1.f - b1) * gi;
        const float vi = b2 * vo + (1.f - b2) * gi * gi;
        m[t] = mi;
        v[t] = vi;
        const float wi = wo - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        w[t] = wi;
        const bf16 h = __float2bfloat16_rn(wi);
        wb[t] = h;
        return h;
    };
    float gi[4], mi[4], vi[4], wi[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int co = co0 + warp + 8 * r;
        if (co >= cout || k0 + lane >= K) continue;
        const long long t = tab.off[k] + (long long)co * K + k0 + lane;
        gi[r] = g[t];
        mi[r] = m[t];
        vi[r] = v[t];
        wi[r] = w[t];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int co = co0 + warp + 8 * r;
        if (co >= cout || k0 + lane >= K) continue;
        sm[lane][warp + 8 * r] =
            step(tab.off[k] + (long long)co * K + k0 + lane, gi[r], mi[r], vi[r], wi[r]);
    }
    // biases and head: stored after a convolution's weights, and last
    if (k0 == 0 && warp == 0 && co0 + lane < cout) {
        const long long t = tab.off[k] + (long long)cout * K + co0 + lane;
        step(t, g[t], m[t], v[t], w[t]);
    }
    if (blockIdx.x == 0 && warp >= 4)
        for (long long t = n - nhead + threadIdx.x - 128; t < n; t += 128) step(t, g[t], m[t], v[t], w[t]);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int kk = k0 + warp + 8 * r;
        if (kk >= K || co0 + lane >= cout) continue;
        const int tap = kk / cin, ci = kk - tap * cin;
        wd[tab.off[k] + ((long long)ci * 9 + tap) * cout + co0 + lane] = sm[warp + 8 * r][lane];
    }
}

// the BF16 copies of every parameter (after the FP32 masters were set)
__global__ void k_bf16_copies(const float* w, long long n, bf16* wb, bf16* wd,
                              const ConvTable tab) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        store_bf16_copies(t, w[t], wb, wd, tab);
}


// how a convolution runs on k_conv_march: cb blocks of kb operand channels, bn output columns per
// CTA; kb = 0: it does not
struct March {
    int kb = 0, cb = 0, bn = 0;
};

struct Conv {
    int src1, C1, up1;  // source tensor index, channels, stored at half resolution
    int src2, C2;       // second source (-1: none)
    int Cout, out;      // output tensor index
    int H, W;           // output resolution
    size_t w_off, b_off;  // offsets into the parameter vector
    // tensor maps of the TMA-fed forward (f) and data-gradient (d) GEMMs: A source 1, A source
    // 2 (concatenation), B; f_ks, d_ks: the K elements per stage of those maps (64 or 32), 0
    // when the shapes do not allow it and the loaders gather with cp.async
    int f_ks = 0, d_ks = 0;
    CUtensorMap fmap[4] = {}, dmap[4] = {};  // [3]: B as 32-row boxes
    // weight gradient (w): A sources 1 and 2 and the output gradient, boxes of 32 channels x 64
    // pixels; w_tma false: gathered with cp.async
    bool w_tma = false;
    CUtensorMap wmap[3] = {};
    // weight gradient from staged rows (k_wgrad_rows): channel blocks of sources 1 and 2 (xb = 0: not
    // so), cb of them per CTA, blocks yb of the output gradient; maps: source 1, 2, dY
    int wr_xb = 0, wr_yb = 0, wr_cb = 0;
    CUtensorMap wrmap[3] = {};
    // forward (fm) and data gradient (dm) on k_conv_march; maps: source 1 (dY for dm) and source 2
    // as boxes of one row of 136 pixels x kb channels, the weights as kb x bn blocks
    March fm, dm;
    CUtensorMap fmmap[3] = {}, dmmap[3] = {};
    // training: gradient with respect to the pre-activation (BF16), the bias gradient's per-block
    // sums, and the event after which the side stream may read them
    bf16* g = nullptr;
    float* bpart = nullptr;
    cudaEvent_t ready = nullptr;
};

struct Tensor {
    int H, W, C;
    bf16* y = nullptr;   // activation
    float* dy = nullptr; // gradient, where it is stored (gradient_buffers: shared in turn)
};

}  // namespace
}  // namespace sg
}  // namespace lbm

using namespace lbm::sg;

struct lbm_surrogate {
    int H = 0, W = 0, base = 0, maxB = 0, device = 0, sms = 152;
    // main stream, and a side stream for the weight and bias gradients of the backward pass, which
    // nothing in the chain of data gradients waits for
    cudaStream_t stream = nullptr, side = nullptr;
    cudaEvent_t head_ready = nullptr, side_done = nullptr;
    std::vector<Tensor> t;      // 0: input (8 channels)
    std::vector<void*> memory;  // the device allocations that everything below points into
    std::vector<Conv> convs;
    std::vector<std::pair<int, int>> pools;  // (from, to)
    int head_in = -1;
    size_t head_w = 0, head_b = 0;
    size_t nparams = 0;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    bf16* wb = nullptr;
    bf16* wbd = nullptr;        // per convolution [C_in][tap][C_out] (data-gradient operand)
    bf16* col = nullptr;      // im2col columns of one layer, where some weight gradient needs them
    float* phi = nullptr;   // head output
    float* hpart = nullptr;
    float* dz = nullptr;      // head: gradient with respect to the pre-sigmoid value, per pixel
    int* n_mask = nullptr;    // loss pixels of the current step
    float *host_loss = nullptr, *host_loss_dev = nullptr;  // mapped host memory
    float *splitk = nullptr, *splitk_side = nullptr;  // split-K partials, one per stream
    size_t splitk_elems = 0;
    int part_blocks = 608;  // head: two resident waves of two blocks per SM
    ConvTable tab{};  // convolution weight shapes for the BF16 copies
    long long adam_t = 0;
    std::string err;
};

extern "C" void lbm_surrogate_destroy(lbm_surrogate* s);

namespace {

lbm_status sfail(lbm_surrogate* s, lbm_status st, const std::string& msg) {
    // reported once (see fail in lbm_api.cu)
    if (st == LBM_ERR_CUDA) cudaGetLastError();
    if (s)
        s->err = msg;
    else
        lbm::set_global_error(msg);
    return st;
}

#define SCUDA(s, expr)                                                                      \
    do {                                                                                    \
        cudaError_t e_ = (expr);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return sfail((s), LBM_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// Latched timeout flag of the tensor-core GEMM: mapped host memory that the kernels write on
// a wait that ran out; reported (and cleared) by the next host call that checks it.
struct TcFlag {
    volatile int* host = nullptr;
    int* dev = nullptr;
};

TcFlag& tc_flag() {
    static std::mutex mu;
    static TcFlag f;
    std::lock_guard<std::mutex> lk(mu);
    if (!f.host) {
        int* h = nullptr;
        if (cudaHostAlloc((void**)&h, sizeof(int), cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            return f;
        }
        *h = 0;
        int* d = nullptr;
        if (cudaHostGetDevicePointer((void**)&d, h, 0) != cudaSuccess) {
            cudaGetLastError();
            cudaFreeHost(h);
            return f;
        }
        f.host = h;
        f.dev = d;
    }
    return f;
}

// true (and the flag cleared) if a tensor-core GEMM launched earlier gave up waiting
bool tc_timed_out() {
    TcFlag& f = tc_flag();
    if (!f.host) return false;
    const bool t = *f.host != 0;
    *f.host = 0;
    return t;
}

template <int BN, int STAGES, bool AMN, bool BMN, bool GA, bool GD, bool GAM, int TMA = 0>
cudaError_t launch_tc(cudaStream_t st, const GemmArgs& a, int splits,
                      const CUtensorMap* maps = nullptr) {
    using TS = lbm::sgtc::TcShape<BN, STAGES, BMN, lbm::sgtc::slice_k(TMA)>;
    // the shared-memory opt-in is per device: one bit per device ordinal that has it (setting it
    // twice from racing host threads is harmless)
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(lbm::sgtc::k_gemm_tc<BN, STAGES, AMN, BMN, GA, GD, GAM, TMA>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, TS::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    int* flag = tc_flag().dev;
    if (!flag) return cudaErrorMemoryAllocation;
    dim3 grid((a.N + BN - 1) / BN, (a.M + lbm::sgtc::BM - 1) / lbm::sgtc::BM, splits);
    static const CUtensorMap none[3] = {};
    const CUtensorMap* m = maps ? maps : none;
    return launch_pdl(lbm::sgtc::k_gemm_tc<BN, STAGES, AMN, BMN, GA, GD, GAM, TMA>, grid,
                      lbm::sgtc::TC_THREADS, TS::SMEM_BYTES, st, a, flag, m[0], m[1], m[2]);
}

// C = A B on the tcgen05 tensor cores, each operand K-major or MN-major (AMN, BMN). The N tile
// is the compiled width that covers N with the fewest computed columns (ties: fewer tiles);
// wide tiles keep two stages so that two CTAs share an SM and one's epilogue overlaps the
// other's MMAs. GA / GAM: A (K-major / MN-major) is the implicit im2col of a.conv; GD: A is the
// gathered data-gradient operand a.dg.
int pick_bn(int N) {
    static const int widths[] = {32, 64, 80, 128, 144, 192, 256};
    int best = 256, best_cols = 1 << 30, best_tiles = 1 << 30;
    for (int w : widths) {
        const int tiles = (N + w - 1) / w, cols = tiles * w;
        if (cols < best_cols || (cols == best_cols && tiles < best_tiles)) {
            best = w;
            best_cols = cols;
            best_tiles = tiles;
        }
    }
    return best;
}

template <bool AMN, bool BMN, bool GA = false, bool GD = false, bool GAM = false>
cudaError_t gemm_tc(cudaStream_t st, const GemmArgs& a, int splits = 1) {
    switch (pick_bn(a.N)) {
        case 32: return launch_tc<32, 3, AMN, BMN, GA, GD, GAM>(st, a, splits);
        case 64: return launch_tc<64, 3, AMN, BMN, GA, GD, GAM>(st, a, splits);
        case 80: return launch_tc<80, 4, AMN, BMN, GA, GD, GAM>(st, a, splits);
        case 128: return launch_tc<128, 3, AMN, BMN, GA, GD, GAM>(st, a, splits);
        case 144: return launch_tc<144, 2, AMN, BMN, GA, GD, GAM>(st, a, splits);
        case 192: return launch_tc<192, 2, AMN, BMN, GA, GD, GAM>(st, a, splits);
        default: return launch_tc<256, 2, AMN, BMN, GA, GD, GAM>(st, a, splits);
    }
}

// cuTensorMapEncodeTiled from the driver (null if the driver does not provide it)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// Map of an NHWC BF16 tensor [N][H][W][C] (C innermost), box ks channels x bw x bh pixels x 1
// image, ks = 64 with 128-byte, 32 with 64-byte, 16 with 32-byte swizzle or 8 without (the K-major
// layouts the MMAs read), out-of-range elements zero.
bool map_nhwc(CUtensorMap* m, const void* base, int C, int W, int H, int N, int bw, int bh,
              int ks, int step = 1, int ystep = 0) {
    const EncodeTiledFn enc = encode_tiled();
    if (!enc) return false;
    const cuuint64_t dim[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    const cuuint64_t stride[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2,
                                  (cuuint64_t)H * W * C * 2};
    // step 2: every second pixel in x and y (the box spans 2 bw x 2 bh pixels, loads bw x bh); ystep:
    // another step in y
    if (!ystep) ystep = step;
    const cuuint32_t box[4] = {(cuuint32_t)ks, (cuuint32_t)(bw * step), (cuuint32_t)(bh * ystep), 1};
    const cuuint32_t es[4] = {1, (cuuint32_t)step, (cuuint32_t)ystep, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dim, stride, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE,
               ks == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
               : ks == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
               : ks == 16 ? CU_TENSOR_MAP_SWIZZLE_32B
                          : CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Map of a row-major BF16 matrix [rows][K], box ks (K) x box_rows, swizzled as in map_nhwc.
bool map_rows(CUtensorMap* m, const void* base, int K, int rows, int box_rows, int ks) {
    const EncodeTiledFn enc = encode_tiled();
    if (!enc) return false;
    const cuuint64_t dim[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t stride[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)ks, (cuuint32_t)box_rows};
    const cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dim, stride, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE,
               ks == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
               : ks == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
               : ks == 16 ? CU_TENSOR_MAP_SWIZZLE_32B
                          : CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// CTAs of a launch up to which gemm_tc_tma takes its narrow, deep form: with it a forward pass of one
// 256 x 256 sample (base 32) takes 284 us, without it 304. Launches of more CTAs hide their slices'
// latency behind one another and would only read the A rows of a tile once per 32 columns (with 304
// instead of 128 the forward pass of one sample takes 297 us, of eight 940 instead of 457).
constexpr long long kFewTiles = 128;

// The TMA-fed gathering GEMM (GA or GD with tensor maps, see Conv::fmap / dmap), ks elements
// of K per stage: N tiles of 32, 64, 128 or 256 columns; few stages, so that several CTAs share
// an SM (each CTA's load latency overlaps the others' MMAs and epilogues).
template <bool GA, bool GD>
cudaError_t gemm_tc_tma(cudaStream_t st, const GemmArgs& a, int splits, const CUtensorMap* maps,
                        int ks) {
    const int bn = pick_bn(a.N);
    // Few tiles: the launch is one chain of slices per CTA, each waiting for its copies. Then every
    // tile is cut into columns of 32 (the same products in the same order) until the SMs are
    // filled, and a CTA keeps eight slices in flight instead of two or three. maps[3]: the weights
    // as 32-row boxes.
    const long long ctas = (long long)((a.N + bn - 1) / bn) * ((a.M + lbm::sgtc::BM - 1) / lbm::sgtc::BM) * splits;
    if (ctas <= kFewTiles && a.N % 32 == 0) {
        const CUtensorMap m[3] = {maps[0], maps[1], maps[3]};
        if (ks == 64) return launch_tc<32, 8, false, false, GA, GD, false, 64>(st, a, splits, m);
        if (ks == 32) return launch_tc<32, 12, false, false, GA, GD, false, 32>(st, a, splits, m);
    }
    if (ks == 64) switch (bn) {
            case 32: return launch_tc<32, 3, false, false, GA, GD, false, 64>(st, a, splits, maps);
            case 64: return launch_tc<64, 3, false, false, GA, GD, false, 64>(st, a, splits, maps);
            case 128: return launch_tc<128, 3, false, false, GA, GD, false, 64>(st, a, splits, maps);
            case 256: return launch_tc<256, 2, false, false, GA, GD, false, 64>(st, a, splits, maps);
            default: break;
        }
    if (ks == 32) switch (bn) {
            case 32: return launch_tc<32, 4, false, false, GA, GD, false, 32>(st, a, splits, maps);
            case 64: return launch_tc<64, 4, false, false, GA, GD, false, 32>(st, a, splits, maps);
            case 128: return launch_tc<128, 6, false, false, GA, GD, false, 32>(st, a, splits, maps);
            case 256: return launch_tc<256, 4, false, false, GA, GD, false, 32>(st, a, splits, maps);
            default: break;
        }
    return cudaErrorInvalidValue;
}

// The gathering GEMMs (GA: forward convolution, GD: data gradient) with fewer output tiles than
// about three quarters of the SMs (the coarse levels): K is cut into up to 2 x 152 / tiles ranges
// of whole 64-wide slices, at least four each, whose FP32 partials k_splitk_finish sums in a
// fixed order before applying the GEMM's own epilogue (bias, leaky ReLU, BF16 or accumulated
// FP32 stores). Otherwise one launch as usual.
template <bool GA, bool GD>
cudaError_t gemm_tc_split(cudaStream_t st, const GemmArgs& a, float* scratch,
                          size_t scratch_elems, const CUtensorMap* maps = nullptr, int ks = 0) {
    const int bn = pick_bn(a.N);
    const long long tiles =
        (long long)((a.N + bn - 1) / bn) * ((a.M + lbm::sgtc::BM - 1) / lbm::sgtc::BM);
    const int nkt = (a.K + lbm::sgtc::BK - 1) / lbm::sgtc::BK;
    long long splits = 1;
    if (tiles < 114 && a.N % 4 == 0 && !a.tout && !a.kchunk && !a.rperm)
        splits = std::min<long long>(2 * 152 / tiles, nkt / 4);
    while (splits > 1 && (size_t)splits * a.M * a.N > scratch_elems) --splits;
    if (splits <= 1)
        return ks ? gemm_tc_tma<GA, GD>(st, a, 1, maps, ks) : gemm_tc<false, false, GA, GD>(st, a);
    const int chunk = (int)((nkt + splits - 1) / splits) * lbm::sgtc::BK;
    const int nsp = (a.K + chunk - 1) / chunk;
    GemmArgs p = a;
    p.Cf = scratch;
    p.Cb = nullptr;
    p.Cf2 = nullptr;
    p.ldc = a.N;
    p.ldc2 = 0;
    p.nsplit = 0;
    p.bias = nullptr;
    p.relu = 0;
    p.accumulate = 0;
    p.kchunk = chunk;
    p.split_stride = (long long)a.M * a.N;
    cudaError_t e = ks ? gemm_tc_tma<GA, GD>(st, p, nsp, maps, ks)
                       : gemm_tc<false, false, GA, GD>(st, p, nsp);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_splitk_finish, dim3(blocks_for((long long)a.M * a.N / 4)), kT, 0, st, scratch,
                      nsp, a.M, a.N, a.bias, a.relu, a.Cb, a.Cf, a.ldc, a.Cf2, a.ldc2, a.nsplit,
                      a.accumulate);
}

// AK / BK: operand stored K-major (else MN-major)
template <bool AK, bool BK>
cudaError_t gemm(cudaStream_t st, const GemmArgs& a) {
    return gemm_tc<!AK, !BK>(st, a);
}

// Weight-gradient GEMM dW[co][k] = sum_p dY[p][co] col[p][k] (K = pixels, both operands
// MN-major): few output tiles and a very long K, so K is split over up to 128 CTA slices whose
// FP32 partials are summed in a fixed order. gather: computed transposed, dW^T = col^T dY with
// the im2col columns gathered by the loader as the 128-row operand (each thread decodes its tap
// and channel once) and stored transposed; else from the im2col buffer a.B.
// The TMA-fed weight gradient (gathered and transposed, maps: Conv::wmap): N tiles of 32, 64,
// 128 or 256 columns, few stages as in gemm_tc_tma.
cudaError_t gemm_wgrad_tma(cudaStream_t st, const GemmArgs& a, int splits, const CUtensorMap* maps) {
    switch (pick_bn(a.N)) {
        case 32: return launch_tc<32, 3, true, true, false, false, true, 1>(st, a, splits, maps);
        case 64: return launch_tc<64, 3, true, true, false, false, true, 1>(st, a, splits, maps);
        case 128: return launch_tc<128, 3, true, true, false, false, true, 1>(st, a, splits, maps);
        case 256: return launch_tc<256, 2, true, true, false, false, true, 1>(st, a, splits, maps);
        default: return cudaErrorInvalidValue;
    }
}

// Launch of k_wgrad_rows: split-K ranges for one wave of CTAs over all column blocks, as far as the
// partials fit `scratch`; the partials are summed in order. a: M = 9 C_in, N = C_out, K = pixels.
cudaError_t sum_splits(cudaStream_t st, const float* part, int splits, long long stride, float* out);
template <int XB, int YB, int CB, bool UP>
cudaError_t launch_wgrad_rows(cudaStream_t st, GemmArgs a, float* scratch, size_t scratch_elems,
                              float* out, const CUtensorMap* maps) {
    using WS = lbm::sgtc::WgradShape<XB, YB, CB, UP>;
    auto* kern = lbm::sgtc::k_wgrad_rows<XB, YB, CB, UP>;
    static std::atomic<unsigned long long> configured{0};
    static std::atomic<int> sms{152};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        int n = 152;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, WS::SMEM);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        sms.store(n);
        configured.fetch_or(bit);
    }
    int* flag = tc_flag().dev;
    if (!flag) return cudaErrorMemoryAllocation;
    const long long stride = (long long)a.N * a.ldc;
    const int groups = (a.conv.C1 + a.conv.C2) / (XB * CB) * (a.N / YB);
    a.K /= 64 * WS::RA * (UP ? 2 : 1);  // slices
    long long splits = std::max(1, std::min(a.K / 2, WS::CTAS * sms.load() / groups));
    splits = std::max(1ll, std::min(splits, (long long)scratch_elems / stride));
    a.kchunk = (int)((a.K + splits - 1) / splits);
    splits = (a.K + a.kchunk - 1) / a.kchunk;
    a.split_stride = splits > 1 ? stride : 0;
    a.Cf = splits > 1 ? scratch : out;
    e = launch_pdl(kern, dim3((unsigned)splits, groups), lbm::sgtc::TC_THREADS, WS::SMEM, st, a, flag,
                   maps[0], maps[1], maps[2]);
    return e != cudaSuccess || splits == 1 ? e : sum_splits(st, scratch, (int)splits, stride, out);
}

cudaError_t gemm_wgrad_rows(cudaStream_t st, const GemmArgs& a, float* scratch, size_t elems, float* out,
                            int xb, int yb, int cb, const CUtensorMap* maps) {
    const int key = xb * 1000 + yb * 10 + cb;
    if (a.conv.up1) switch (key) {
            case 32161: return launch_wgrad_rows<32, 16, 1, true>(st, a, scratch, elems, out, maps);
            case 32322: return launch_wgrad_rows<32, 32, 2, true>(st, a, scratch, elems, out, maps);
            default: return cudaErrorInvalidValue;
        }
    switch (key) {
        case 16161: return launch_wgrad_rows<16, 16, 1, false>(st, a, scratch, elems, out, maps);
        case 16162: return launch_wgrad_rows<16, 16, 2, false>(st, a, scratch, elems, out, maps);
        case 16321: return launch_wgrad_rows<16, 32, 1, false>(st, a, scratch, elems, out, maps);
        case 32321: return launch_wgrad_rows<32, 32, 1, false>(st, a, scratch, elems, out, maps);
        case 32322: return launch_wgrad_rows<32, 32, 2, false>(st, a, scratch, elems, out, maps);
        default: return cudaErrorInvalidValue;
    }
}

// out = the sum of `splits` FP32 partials of `stride` values each, in split order
cudaError_t sum_splits(cudaStream_t st, const float* part, int splits, long long stride, float* out) {
    if (stride % 4 == 0 && ((uintptr_t)out & 15) == 0)
        return launch_pdl(k_splitk_sum4, dim3((unsigned)((stride / 4 + 31) / 32)), splits < 64 ? 256 : 1024,
                          0, st, part, splits, stride, stride, out);
    return launch_pdl(k_splitk_sum, dim3(blocks_for(stride)), kT, 0, st, part, splits, stride, stride,
                      out);
}

// How a convolution runs on k_conv_march: blocks of kb channels, cb of them, bn output columns per
// CTA; kb = 0: it does not. Maps: source 1 (dY for the data gradient) and source 2 as boxes of one
// row of 136 pixels x kb channels, weights as kb x bn blocks. parts: how many partial sums per column a
// fused leaky-ReLU adjoint (GemmArgs::rg) left, 0 when it was not fused.
template <int KB, int CB, int BN, bool GD, bool UP>
cudaError_t launch_march(cudaStream_t st, GemmArgs a, const CUtensorMap* maps, int* parts) {
    using MS = lbm::sgtc::MarchShape<KB, CB, BN, GD, UP>;
    auto* kern = lbm::sgtc::k_conv_march<KB, CB, BN, GD, UP>;
    static std::atomic<unsigned long long> configured{0};
    static std::atomic<int> sms{152};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        int n = 152;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, MS::SMEM);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        sms.store(n);
        configured.fetch_or(bit);
    }
    int* flag = tc_flag().dev;
    if (!flag) return cudaErrorMemoryAllocation;
    const int H = GD ? a.dg.H : a.conv.H, W = GD ? a.dg.W : a.conv.W;
    const int rh = UP ? H / 2 : H, rw = UP ? W / 2 : W, nb = a.N / BN;
    const long long image = MS::UD ? (long long)rh * rw : (long long)H * W;  // rows of the GEMM
    const int strips = (int)(a.M / image) * (rw / 128);
    // one wave of CTAs: chunks of rows so that strips x chunks x column blocks fill the SMs
    const int want = std::max(1, MS::PER_SM * sms.load() / std::max(1, strips * nb));
    const int chunk = std::max(1, (rh + want - 1) / want);
    const dim3 grid((unsigned)strips * ((rh + chunk - 1) / chunk), nb);
    if (grid.x > (unsigned)kReluBlocks) a.rg = nullptr;  // rpart's columns
    if (GD && !a.rg && !a.Cf) return cudaErrorInvalidValue;  // (fused_always rules this out)
    if (parts) *parts = a.rg ? (int)grid.x : 0;
    return launch_pdl(kern, grid, lbm::sgtc::MARCH_THREADS, MS::SMEM, st, a, flag, maps[0], maps[1],
                      maps[2], chunk);
}

// The first convolution on k_conv0 / k_wgrad0: rows a multiple of 128 pixels, 16 or 32 outputs and an
// input the copy engine can address (the maps are made per call, x being the caller's).
bool conv0_ok(const Conv& c, const void* x) {
    return c.C1 == 8 && c.C2 == 0 && !c.up1 && c.W % 128 == 0 && (c.Cout == 16 || c.Cout == 32) &&
           ((uintptr_t)x & 15) == 0;
}

template <int N>
cudaError_t launch_conv0(cudaStream_t st, const GemmArgs& a, const CUtensorMap& mx) {
    int* flag = tc_flag().dev;
    if (!flag) return cudaErrorMemoryAllocation;
    const unsigned ctas = (unsigned)(a.M / (128 * lbm::sgtc::C0_ROWS));
    return launch_pdl(lbm::sgtc::k_conv0<N>, dim3(ctas), lbm::sgtc::TC_THREADS,
                      lbm::sgtc::Conv0Shape<N>::SMEM, st, a, flag, mx);
}

template <int N>
cudaError_t launch_wgrad0(cudaStream_t st, GemmArgs a, float* scratch, float* out, const CUtensorMap& mx,
                          const CUtensorMap& mdy) {
    using WS = lbm::sgtc::Wgrad0Shape<N>;
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(lbm::sgtc::k_wgrad0<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 WS::SMEM);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    int* flag = tc_flag().dev;
    if (!flag) return cudaErrorMemoryAllocation;
    // K ranges of at least four slices, at most two per SM
    const int slices = a.K / 128;
    int splits = std::max(1, std::min(304, slices / 4));
    const int per = (slices + splits - 1) / splits;
    splits = (slices + per - 1) / per;
    const long long stride = (long long)N * 72;
    a.kchunk = per * 128;
    a.split_stride = splits > 1 ? stride : 0;
    a.Cf = splits > 1 ? scratch : out;
    e = launch_pdl(lbm::sgtc::k_wgrad0<N>, dim3(splits), lbm::sgtc::TC_THREADS, WS::SMEM, st, a, flag, mx,
                   mdy);
    return e != cudaSuccess || splits == 1 ? e : sum_splits(st, scratch, splits, stride, out);
}

template <bool GD>
cudaError_t conv_march(cudaStream_t st, const GemmArgs& a, const March& m, const CUtensorMap* maps,
                       int* parts = nullptr) {
    const int key = m.kb * 1000 + m.cb * 100 + m.bn;
    if constexpr (!GD) {
        if (a.conv.up1) switch (key) {
                case 32116: return launch_march<32, 1, 16, false, true>(st, a, maps, parts);
                case 32232: return launch_march<32, 2, 32, false, true>(st, a, maps, parts);
                default: return cudaErrorInvalidValue;
            }
    } else if (a.dg.up1) {
        switch (key) {
            case 16132: return launch_march<16, 1, 32, true, true>(st, a, maps, parts);
            case 32164: return launch_march<32, 1, 64, true, true>(st, a, maps, parts);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (key) {
        case 16116: return launch_march<16, 1, 16, GD, false>(st, a, maps, parts);
        case 16132: return launch_march<16, 1, 32, GD, false>(st, a, maps, parts);
        // forward only (two sources of 16 channels), data gradient only (32 outputs of 16 inputs)
        case GD ? 32116 : 16216: return launch_march<GD ? 32 : 16, GD ? 1 : 2, 16, GD, false>(st, a, maps, parts);
        case 32132: return launch_march<32, 1, 32, GD, false>(st, a, maps, parts);
        case 32164: return launch_march<32, 1, 64, GD, false>(st, a, maps, parts);
        case 32232: return launch_march<32, 2, 32, GD, false>(st, a, maps, parts);
        case 32264: return launch_march<32, 2, 64, GD, false>(st, a, maps, parts);
        default: return cudaErrorInvalidValue;
    }
}
// the forms conv_march has
bool march_form(const March& m, bool gd, bool up) {
    const int key = m.kb * 1000 + m.cb * 100 + m.bn;
    if (up) return gd ? key == 16132 || key == 32164 : key == 32116 || key == 32232;
    return key == 16116 || key == 16132 || key == (gd ? 32116 : 16216) || key == 32132 || key == 32164 ||
           key == 32232 || key == 32264;
}

cudaError_t gemm_wgrad(cudaStream_t st, GemmArgs a, float* scratch, size_t scratch_elems,
                       float* out, bool gather, const CUtensorMap* maps = nullptr) {
    if (gather) {
        // rows: the 9 C_in im2col columns; columns: C_out; a.ldc (= 9 C_in) stays the row
        // length of dW, written at dW[n * ldc + m]
        GemmArgs t = a;
        t.M = a.N;
        t.N = a.M;
        t.B = a.A;
        t.ldb = a.lda;
        t.tout = 1;
        a = t;
    }
    // enough K slices for every SM to hold as many CTAs as fit (three of the narrow tiles, two
    // of the wide ones): each CTA keeps only two K-slices of gathers in flight
    const int bn = pick_bn(a.N);
    const int tiles = ((a.N + bn - 1) / bn) * ((a.M + lbm::sgtc::BM - 1) / lbm::sgtc::BM);
    const int occ = bn <= 64 && !maps ? 3 : 2;
    int splits = std::max(1, std::min(128, occ * 152 / std::max(1, tiles)));
    const long long stride = gather ? (long long)a.N * a.ldc : (long long)a.M * a.ldc;
    while (splits > 1 && (size_t)splits * stride > scratch_elems) splits /= 2;
    if (splits == 1) {
        a.Cf = out;
        return maps     ? gemm_wgrad_tma(st, a, 1, maps)
               : gather ? gemm_tc<true, true, false, false, true>(st, a)
                        : gemm_tc<true, true>(st, a);
    }
    int chunk = (a.K + splits - 1) / splits;
    chunk = (chunk + lbm::sgtc::BK - 1) / lbm::sgtc::BK * lbm::sgtc::BK;
    splits = (a.K + chunk - 1) / chunk;
    a.Cf = scratch;
    a.kchunk = chunk;
    a.split_stride = stride;
    cudaError_t e = maps     ? gemm_wgrad_tma(st, a, splits, maps)
                    : gather ? gemm_tc<true, true, false, false, true>(st, a, splits)
                             : gemm_tc<true, true>(st, a, splits);
    if (e != cudaSuccess) return e;
    return sum_splits(st, scratch, splits, stride, out);
}

// BF16 copies of the weights (after the FP32 masters changed): W for the forward pass and the
// weight gradient, the rearranged copy for the data gradient
cudaError_t refresh_bf16_weights(lbm_surrogate* s) {
    k_bf16_copies<<<blocks_for((long long)s->nparams), kT, 0, s->stream>>>(
        s->w, (long long)s->nparams, s->wb, s->wbd, s->tab);
    return cudaGetLastError();
}

int ilog2_exact(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return (1 << l) == v ? l : -1;
}

PixDims pix_dims(int H, int W) { return PixDims{H, W, ilog2_exact(H), ilog2_exact(W)}; }

// im2col of convolution c (channel groups of 8, a power of two, checked at creation)
cudaError_t launch_im2col(lbm_surrogate* s, cudaStream_t st, const Conv& c, int B) {
    const bf16* x1 = s->t[c.src1].y;
    const bf16* x2 = c.src2 >= 0 ? s->t[c.src2].y : nullptr;
    const PixDims d = pix_dims(c.H, c.W);
    const int P = B * c.H * c.W;
    const int lc8 = ilog2_exact((c.C1 + c.C2) / 8);
    const long long total = (long long)P * 9 * ((c.C1 + c.C2) / 8);
    return launch_pdl(d.lh >= 0 && d.lw >= 0 ? k_im2col<true> : k_im2col<false>,
                      dim3(blocks_for(total)), kT, 0, st, x1, c.C1, c.up1, x2, c.C2, d, P, lc8, s->col);
}

int add_tensor(lbm_surrogate* s, int H, int W, int C) {
    Tensor x;
    x.H = H;
    x.W = W;
    x.C = C;
    s->t.push_back(x);
    return (int)s->t.size() - 1;
}

int add_conv(lbm_surrogate* s, int src1, int up1, int src2, int Cout) {
    Conv c;
    c.src1 = src1;
    c.C1 = s->t[src1].C;
    c.up1 = up1;
    c.src2 = src2;
    c.C2 = src2 >= 0 ? s->t[src2].C : 0;
    c.H = up1 ? s->t[src1].H * 2 : s->t[src1].H;
    c.W = up1 ? s->t[src1].W * 2 : s->t[src1].W;
    c.Cout = Cout;
    c.out = add_tensor(s, c.H, c.W, Cout);
    c.w_off = s->nparams;
    s->nparams += (size_t)Cout * 9 * (c.C1 + c.C2);
    c.b_off = s->nparams;
    s->nparams += Cout;
    s->convs.push_back(c);
    return c.out;
}

void build(lbm_surrogate* s) {
    const int b = s->base;
    int x = add_tensor(s, s->H, s->W, 8);
    int s1 = add_conv(s, add_conv(s, x, 0, -1, b), 0, -1, b);
    int p1 = add_tensor(s, s->H / 2, s->W / 2, b);
    s->pools.push_back({s1, p1});
    int s2 = add_conv(s, add_conv(s, p1, 0, -1, 2 * b), 0, -1, 2 * b);
    int p2 = add_tensor(s, s->H / 4, s->W / 4, 2 * b);
    s->pools.push_back({s2, p2});
    int s3 = add_conv(s, add_conv(s, p2, 0, -1, 4 * b), 0, -1, 4 * b);
    int p3 = add_tensor(s, s->H / 8, s->W / 8, 4 * b);
    s->pools.push_back({s3, p3});
    int bt = add_conv(s, add_conv(s, p3, 0, -1, 8 * b), 0, -1, 8 * b);
    int u3 = add_conv(s, bt, 1, -1, 4 * b);
    int d3 = add_conv(s, add_conv(s, u3, 0, s3, 4 * b), 0, -1, 4 * b);
    int u2 = add_conv(s, d3, 1, -1, 2 * b);
    int d2 = add_conv(s, add_conv(s, u2, 0, s2, 2 * b), 0, -1, 2 * b);
    int u1 = add_conv(s, d2, 1, -1, b);
    int d1 = add_conv(s, add_conv(s, u1, 0, s1, b), 0, -1, b);
    s->head_in = d1;
    s->head_w = s->nparams;
    s->nparams += b;
    s->head_b = s->nparams;
    s->nparams += 1;
}

// The convolution whose output is c's first source, when c alone reads that output (no pool, no other
// convolution, not the head) and its channels come in the 16s of k_conv_march's epilogue; else null.
const Conv* sole_producer(const lbm_surrogate* s, const Conv& c) {
    const Conv* p = nullptr;
    int readers = c.src1 == s->head_in;
    for (const Conv& o : s->convs) {
        if (o.out == c.src1) p = &o;
        readers += (o.src1 == c.src1) + (o.src2 == c.src1);
    }
    for (const auto& pl : s->pools) readers += pl.first == c.src1;
    return readers == 1 && c.C1 % 16 == 0 ? p : nullptr;
}

// True when every training step forms the pre-activation gradient of c's first source in the epilogue of c's
// data gradient (launch_march has at most max(strips, two per SM) CTAs along its rows), so that the
// source's FP32 gradient is never stored.
bool fused_always(const lbm_surrogate* s, const Conv& c) {
    const long long strips = (long long)s->maxB * ((c.up1 ? c.W / 2 : c.W) / 128);
    return c.dm.kb && sole_producer(s, c) && std::max<long long>(strips, 2 * s->sms) <= kReluBlocks;
}

struct Part {
    void** p;
    size_t bytes;
};

// Sets every pointer to its part of one allocation (each 256-byte aligned). One by one the 80 parts of a
// small network took longer than everything else in its creation.
cudaError_t allocate(lbm_surrogate* s, const std::vector<Part>& parts) {
    size_t total = 0;
    for (const Part& q : parts) total += (q.bytes + 255) / 256 * 256;
    char* base = nullptr;
    const cudaError_t e = total ? cudaMalloc((void**)&base, total) : cudaSuccess;
    if (e != cudaSuccess) return e;
    if (base) s->memory.push_back(base);
    for (const Part& q : parts) {
        *q.p = base;
        base += (q.bytes + 255) / 256 * 256;
    }
    return cudaSuccess;
}

// Buffers of the FP32 activation gradients (index per tensor, -1: not stored; sizes for max_batch images).
// A gradient lives on the main stream from the first data gradient that writes it to the leaky-ReLU pass
// of its convolution (a pooled map's: of the pool's source), in the order of queue_train_step, so a few
// buffers serve all of them.
std::vector<int> gradient_buffers(const lbm_surrogate* s, const std::vector<char>& stored,
                                  std::vector<size_t>* size) {
    std::vector<int> buf(s->t.size(), -1), free;
    auto release = [&](int t) {
        if (t >= 0 && buf[t] >= 0) free.push_back(buf[t]);
    };
    auto take = [&](int t) {
        if (t < 0 || !stored[t] || buf[t] >= 0) return;
        const Tensor& x = s->t[t];
        const size_t n = (size_t)s->maxB * x.H * x.W * x.C;
        // the largest free buffer (grown if it is too small), else a new one
        auto big = std::max_element(free.begin(), free.end(),
                                    [&](int a, int b) { return (*size)[a] < (*size)[b]; });
        if (big == free.end()) {
            buf[t] = (int)size->size();
            size->push_back(n);
        } else {
            buf[t] = *big;
            (*size)[*big] = std::max((*size)[*big], n);
            free.erase(big);
        }
    };
    for (int ci = (int)s->convs.size() - 1; ci >= 0; --ci) {
        const Conv& c = s->convs[ci];
        release(c.out);
        for (const auto& pl : s->pools)
            if (pl.first == c.out) release(pl.second);
        take(c.src1);
        take(c.src2);
    }
    return buf;
}

// the main stream waits for what the side stream holds so far
cudaError_t join_side(lbm_surrogate* s) {
    const cudaError_t e = cudaEventRecord(s->side_done, s->side);
    return e == cudaSuccess ? cudaStreamWaitEvent(s->stream, s->side_done, 0) : e;
}

// the head on the last activation; with a target (training) also its loss terms and gradients
cudaError_t launch_head(lbm_surrogate* s, int blocks, float* phi, long long P, const float* target,
                        const uint8_t* mask) {
    auto* k = s->base == 32 ? k_head<32> : s->base == 16 ? k_head<16> : k_head<8>;
    return launch_pdl(k, dim3(blocks), kT, 0, s->stream, s->t[s->head_in].y, s->w + s->head_w,
                      s->w + s->head_b, phi, P, target, mask, s->n_mask, s->dz, s->hpart);
}

lbm_status forward(lbm_surrogate* s, const bf16* x, int B) {
    s->t[0].y = const_cast<bf16*>(x);
    // convolutions run in production order; a pool runs right after the conv that feeds it
    for (const Conv& c : s->convs) {
        const Tensor& a = s->t[c.src1];
        if (a.y == nullptr) return sfail(s, LBM_ERR_STATE, "surrogate: missing activation");
        const int Cin = c.C1 + c.C2;
        const long long P = (long long)B * c.H * c.W;
        // implicit GEMM: the 3 x 3 neighbourhoods are gathered from the activations by the
        // tensor-core kernel's loader (no im2col buffer)
        GemmArgs g{};
        g.conv.x1 = a.y;
        g.conv.x2 = c.src2 >= 0 ? s->t[c.src2].y : nullptr;
        g.conv.C1 = c.C1;
        g.conv.C2 = c.C2;
        g.conv.up1 = c.up1;
        g.conv.H = c.H;
        g.conv.W = c.W;
        g.conv.lc = ilog2_exact(Cin);
        g.B = s->wb + c.w_off;
        g.M = (int)P;
        g.N = c.Cout;
        g.K = 9 * Cin;
        g.ldb = 9 * Cin;
        g.Cb = s->t[c.out].y;
        g.ldc = c.Cout;
        g.bias = s->w + c.b_off;
        g.relu = 1;
        if (c.up1 && c.f_ks) g.rperm = std::min(c.W, 128) / 2;
        CUtensorMap mx;
        if (c.src1 == 0 && conv0_ok(c, a.y) &&
            map_nhwc(&mx, a.y, 8, c.W, c.H, B, lbm::sgtc::C0_PITCH, lbm::sgtc::C0_ROWS + 2, 8))
            SCUDA(s, c.Cout == 32 ? launch_conv0<32>(s->stream, g, mx)
                                  : launch_conv0<16>(s->stream, g, mx));
        else if (c.fm.kb)
            SCUDA(s, conv_march<false>(s->stream, g, c.fm, c.fmmap));
        else
            SCUDA(s, (gemm_tc_split<true, false>(s->stream, g, s->splitk, s->splitk_elems, c.fmap,
                                                  c.f_ks)));
        // a pool whose source is this conv's output runs right after it
        for (const auto& pl : s->pools)
            if (pl.first == c.out) {
                const Tensor& src = s->t[pl.first];
                const long long n8 = (long long)B * src.H * src.W / 4 * (src.C / 8);
                SCUDA(s, launch_pdl(k_avgpool, dim3(blocks_for(n8)), kT, 0, s->stream, src.y,
                                    s->t[pl.second].y, n8, src.H, src.W, ilog2_exact(src.C / 8)));
            }
    }
    return LBM_OK;
}

// k_conv_march where it applies: operand rows a multiple of 128 pixels wide (for a forward
// upsampling convolution the half-resolution source's), 16, 32 or 64 operand channels (input, both
// sources' blocks aligned; output gradient), 16, 32 or a multiple of 64 output columns. At most
// 178 KB of shared memory; with 128 operand channels rows and weights would not fit together, so those
// layers keep the boxes per tap.
void make_march_maps(lbm_surrogate* s, Conv& c) {
    auto blocks = [](int c1, int c2, int n) {
        March m;
        const int cin = c1 + c2;
        m.kb = c1 % 32 == 0 && c2 % 32 == 0 ? 32 : c1 % 16 == 0 && c2 % 16 == 0 ? 16 : 0;
        m.cb = m.kb ? cin / m.kb : 0;
        m.bn = n % 64 == 0 ? 64 : n % 32 == 0 ? 32 : n % 16 == 0 ? 16 : 0;
        return m;
    };
    if (c.src1 == 0) return;
    const int cin = c.C1 + c.C2, ow = c.up1 ? c.W / 2 : c.W, oh = c.up1 ? c.H / 2 : c.H;
    if (ow % 128 == 0 && !(c.up1 && c.C2)) {
        const March m = blocks(c.C1, c.C2, c.Cout);
        if (m.kb && m.bn && march_form(m, false, c.up1) &&
            map_nhwc(&c.fmmap[0], s->t[c.src1].y, c.C1, ow, oh, s->maxB, 136, 1, m.kb) &&
            (c.src2 < 0 || map_nhwc(&c.fmmap[1], s->t[c.src2].y, c.C2, ow, oh, s->maxB, 136, 1, m.kb)) &&
            map_rows(&c.fmmap[2], s->wb + c.w_off, 9 * cin, c.Cout, m.bn, m.kb))
            c.fm = m;
    }
    if (ow % 128 == 0 && !(c.up1 && c.C2)) {
        const March m = blocks(c.Cout, 0, cin);
        // a column block of eight lies on one side of the split between the sources; upsampling: every
        // second pixel, in two boxes (a box spans at most 256)
        if (m.kb && m.bn && march_form(m, true, c.up1) && c.C1 % 8 == 0 &&
            (c.up1 ? map_nhwc(&c.dmmap[0], c.g, c.Cout, c.W, c.H, s->maxB, 72, 1, m.kb, 2, 1) &&
                         map_nhwc(&c.dmmap[1], c.g, c.Cout, c.W, c.H, s->maxB, 64, 1, m.kb, 2, 1)
                   : map_nhwc(&c.dmmap[0], c.g, c.Cout, c.W, c.H, s->maxB, 136, 1, m.kb)) &&
            map_rows(&c.dmmap[2], s->wbd + c.w_off, 9 * c.Cout, cin, m.bn, m.kb))
            c.dm = m;
    }
}

// Column blocks (groups of input channels x blocks of output channels) up to which the weight gradient
// runs on k_wgrad_rows: every block reads the operands again, and with more of them the tiles of
// k_gemm_tc are wide enough (64 x 64 x 8: 64 -> 128 channels, 4 blocks, 16 us; 128 -> 128, 8 blocks, 24
// against 21; 256 -> 128, 16 blocks, 40 against 34).
constexpr int kWgradGroups = 4;

// The weight gradient on k_wgrad_rows: rows of the source a multiple of 64 pixels, whole slices of rows,
// channels in blocks of 32 or 16.
void make_wgrad_maps(lbm_surrogate* s, Conv& c) {
    if (c.src1 == 0 || (c.up1 && c.C2)) return;
    const int cin = c.C1 + c.C2, ow = c.up1 ? c.W / 2 : c.W, oh = c.up1 ? c.H / 2 : c.H;
    const int xb = c.C1 % 32 == 0 && c.C2 % 32 == 0 ? 32 : c.C1 % 16 == 0 && c.C2 % 16 == 0 ? 16 : 0;
    const int yb = c.Cout % 32 == 0 ? 32 : c.Cout == 16 ? 16 : 0;
    if (!xb || !yb || ow % 64 || c.H % (xb == 32 ? 2 : 4)) return;
    const int cb = cin / xb % 2 ? 1 : 2, key = xb * 1000 + yb * 10 + cb;
    const bool form = c.up1 ? key == 32161 || key == 32322
                            : key == 16161 || key == 16162 || key == 16321 || key == 32321 || key == 32322;
    if (!form || cin / (xb * cb) * (c.Cout / yb) > kWgradGroups) return;
    const int ra = xb == 32 ? 2 : 4, rows = c.up1 ? 3 : ra + 2;
    if (map_nhwc(&c.wrmap[0], s->t[c.src1].y, c.C1, ow, oh, s->maxB, 72, rows, xb) &&
        (c.src2 < 0 || map_nhwc(&c.wrmap[1], s->t[c.src2].y, c.C2, ow, oh, s->maxB, 72, rows, xb)) &&
        map_nhwc(&c.wrmap[2], c.g, c.Cout, c.W, c.H, s->maxB, 64, ra, yb, c.up1 ? 2 : 1, 1)) {
        c.wr_xb = xb;
        c.wr_yb = yb;
        c.wr_cb = cb;
    }
}

// Tensor maps for the forward and data-gradient GEMMs whose A operand the copy engine can fetch
// as boxes: no upsampled source, channel counts multiples of 64 (one K-slice of 64 = one tap of
// one source) or else of 32 (slices of 32), the 128 rows of a tile a whole block of pixels of
// one image, and N tiles of 32, 64, 128 or 256 columns. The network input (its pointer changes
// per call) never qualifies.
void make_tensor_maps(lbm_surrogate* s) {
    auto tma_width = [](int bn) { return bn == 32 || bn == 64 || bn == 128 || bn == 256; };
    auto slice = [](int a, int b) { return a % 64 == 0 && b % 64 == 0 ? 64
                                         : a % 32 == 0 && b % 32 == 0 ? 32 : 0; };
    for (Conv& c : s->convs) {
        const int W = c.W, H = c.H;
        make_march_maps(s, c);
        make_wgrad_maps(s, c);
        if (c.up1 && c.src1 != 0) {
            // forward of an upsampling convolution: tile rows in runs of even, then odd output
            // columns, each run a box of half a tile row of source pixels
            const int fk = slice(c.C1, c.C2);
            if ((W % 128 == 0 || 128 % W == 0) && (H * W) % 128 == 0 && W >= 16 && fk &&
                c.C2 == 0 && tma_width(pick_bn(c.Cout)) &&
                map_nhwc(&c.fmap[0], s->t[c.src1].y, c.C1, W / 2, H / 2, s->maxB,
                         std::min(W, 128) / 2, 1, fk) &&
                map_rows(&c.fmap[2], s->wb + c.w_off, 9 * c.C1, c.Cout, pick_bn(c.Cout), fk) &&
                map_rows(&c.fmap[3], s->wb + c.w_off, 9 * c.C1, c.Cout, 32, fk))
                c.f_ks = fk;
            // data gradient of an upsampling convolution: rows are source pixels (half
            // resolution), the output gradient read every second pixel; B wraps every 9 Cout
            const int Ws = W / 2, Hs = H / 2, cin = c.C1 + c.C2, dk = slice(c.Cout, 0);
            if ((Ws % 128 == 0 || 128 % Ws == 0) && (Hs * Ws) % 128 == 0 && dk &&
                (9 * c.Cout) % dk == 0 && tma_width(pick_bn(cin))) {
                const int bw = std::min(Ws, 128), bh = 128 / bw;
                if (map_nhwc(&c.dmap[0], c.g, c.Cout, W, H, s->maxB, bw, bh, dk, 2) &&
                    map_rows(&c.dmap[2], s->wbd + c.w_off, 9 * c.Cout, cin, pick_bn(cin), dk) &&
                    map_rows(&c.dmap[3], s->wbd + c.w_off, 9 * c.Cout, cin, 32, dk))
                    c.d_ks = dk;
            }
            // weight gradient: 32 source pixels x 32 channels per box, and 32 output-gradient
            // pixels taken every second one
            if (W % 64 == 0 && c.C2 == 0 && c.C1 % 32 == 0 && c.Cout % 32 == 0 &&
                tma_width(pick_bn(c.Cout)))
                c.w_tma = map_nhwc(&c.wmap[0], s->t[c.src1].y, c.C1, Ws, Hs, s->maxB, 32, 1, 32) &&
                          map_nhwc(&c.wmap[2], c.g, c.Cout, W, H, s->maxB, 32, 1, 32, 2);
            continue;
        }
        if (!((W % 128 == 0 || 128 % W == 0) && (H * W) % 128 == 0) || c.src1 == 0)
            continue;
        const int bw = std::min(W, 128), bh = 128 / bw, cin = c.C1 + c.C2;
        const int fk = slice(c.C1, c.C2), dk = slice(c.Cout, 0);
        if (fk && tma_width(pick_bn(c.Cout)) &&
            map_nhwc(&c.fmap[0], s->t[c.src1].y, c.C1, W, H, s->maxB, bw, bh, fk) &&
            (c.src2 < 0 || map_nhwc(&c.fmap[1], s->t[c.src2].y, c.C2, W, H, s->maxB, bw, bh, fk)) &&
            map_rows(&c.fmap[2], s->wb + c.w_off, 9 * cin, c.Cout, pick_bn(c.Cout), fk) &&
            map_rows(&c.fmap[3], s->wb + c.w_off, 9 * cin, c.Cout, 32, fk))
            c.f_ks = fk;
        if (W % 64 == 0 || 64 % W == 0) {
            const int ww = std::min(W, 64), wh = 64 / ww;
            c.w_tma = c.C1 % 32 == 0 && c.C2 % 32 == 0 && c.Cout % 32 == 0 &&
                      tma_width(pick_bn(c.Cout)) &&
                      map_nhwc(&c.wmap[0], s->t[c.src1].y, c.C1, W, H, s->maxB, ww, wh, 32) &&
                      (c.src2 < 0 ||
                       map_nhwc(&c.wmap[1], s->t[c.src2].y, c.C2, W, H, s->maxB, ww, wh, 32)) &&
                      map_nhwc(&c.wmap[2], c.g, c.Cout, W, H, s->maxB, ww, wh, 32);
        }
        if (dk && tma_width(pick_bn(cin)) &&
            map_nhwc(&c.dmap[0], c.g, c.Cout, W, H, s->maxB, bw, bh, dk) &&
            map_rows(&c.dmap[2], s->wbd + c.w_off, 9 * c.Cout, cin, pick_bn(cin), dk) &&
            map_rows(&c.dmap[3], s->wbd + c.w_off, 9 * c.Cout, cin, 32, dk))
            c.d_ks = dk;
    }
}

// A call that fails while queuing waits for what it queued before it reports: the caller may free or reuse
// the input, target and mask, and the next call's kernels the buffers that the side stream reads.
lbm_status settle(lbm_surrogate* s, lbm_status st) {
    if (st != LBM_OK) {
        cudaStreamSynchronize(s->side);
        cudaStreamSynchronize(s->stream);
    }
    return st;
}

lbm_status queue_forward(lbm_surrogate* s, const bf16* x, int32_t B, float* phi) {
    lbm_status st = forward(s, x, B);
    if (st != LBM_OK) return st;
    const long long P = (long long)B * s->H * s->W;
    const int nb = std::min(s->part_blocks, blocks_for(P));
    SCUDA(s, launch_head(s, nb, phi, P, nullptr, nullptr));
    return LBM_OK;
}

// Queues one training step on the two streams: gradients of the masked MSE into s->g, the loss into
// host_loss; with lr > 0 also an Adam update.
lbm_status queue_train_step(lbm_surrogate* s, const void* xin, const float* target,
                            const uint8_t* mask, int32_t B, float lr) {
    lbm_status st = forward(s, (const bf16*)xin, B);
    if (st != LBM_OK) return st;
    const long long P = (long long)B * s->H * s->W;
    // Everything below is queued without waiting for the device. Activation gradients need no
    // zero fill: the first consumer's data gradient stores, a further one would accumulate.
    SCUDA(s, cudaMemsetAsync(s->n_mask, 0, sizeof(int), s->stream));
    SCUDA(s, launch_pdl(k_mask_count, dim3((unsigned)std::min<long long>(152, blocks_for(P / 16 + 1))),
                        kT, 0, s->stream, mask, P, s->n_mask));
    std::vector<char> written(s->t.size(), 0);
    BiasTable bias{};  // of the layers on the side stream
    // per tensor: the bias gradient's partial sums when its convolution's g is already there
    std::vector<int> fused(s->t.size(), 0);
    const int C = s->base;
    const int nb = std::min(s->part_blocks, blocks_for(P));
    SCUDA(s, launch_head(s, nb, s->phi, P, target, mask));
    // head gradients and loss: sums of the per-block partials (C weights, loss, bias)
    SCUDA(s, cudaEventRecord(s->head_ready, s->stream));
    SCUDA(s, cudaStreamWaitEvent(s->side, s->head_ready, 0));
    SCUDA(s, launch_pdl(k_colsum_final, dim3(C + 2), kT, 0, s->side, s->hpart, nb, C + 2,
                        s->g + s->head_w, 0, s->host_loss_dev));
    // backward through the convolutions (reverse order), pools interleaved
    for (int ci = (int)s->convs.size() - 1; ci >= 0; --ci) {
        const Conv& c = s->convs[ci];
        // gradient arriving at this conv's output also includes the pool path (already added,
        // pools run before: a pool's output gradient is complete once every later conv is done)
        const float* dyp = nullptr;
        for (const auto& pl : s->pools)
            if (pl.first == c.out) dyp = s->t[pl.second].dy;
        Tensor& o = s->t[c.out];
        const int Cin = c.C1 + c.C2;
        const long long Pc = (long long)B * c.H * c.W;
        const long long n_out = Pc * c.Cout;
        // leaky-ReLU adjoint (with the pool's), BF16 copy and the bias gradient's partial sums
        const int rb = fused[c.out] ? fused[c.out]
                                    : (int)std::min<long long>(kReluBlocks, (n_out / 8 + kT - 1) / kT);
        if (fused[c.out]) {
        } else if (c.out == s->head_in)
            SCUDA(s, launch_pdl(k_relu_bias<2>, dim3(rb), kT, 0, s->stream, s->dz, nullptr,
                                s->w + s->head_w, o.y, c.g, n_out / 8, c.Cout, c.H, c.W, c.bpart));
        else
            SCUDA(s, launch_pdl(dyp ? k_relu_bias<1> : k_relu_bias<0>, dim3(rb), kT, 0, s->stream,
                                o.dy, dyp, nullptr, o.y, c.g, n_out / 8, c.Cout, c.H, c.W, c.bpart));
        // the side stream takes the bias and weight gradients from here; the first convolution's
        // stay on the main stream, which has nothing left to do by then
        const bool last = c.src1 == 0;
        cudaStream_t ws = last ? s->stream : s->side;
        if (!last) {
            SCUDA(s, cudaEventRecord(c.ready, s->stream));
            SCUDA(s, cudaStreamWaitEvent(s->side, c.ready, 0));
        }
        if (last) {
            SCUDA(s, launch_pdl(k_colsum_final, dim3(c.Cout), kT, 0, ws, c.bpart, rb, c.Cout,
                                s->g + c.b_off, 1, nullptr));
        } else {
            bias.part[bias.n] = c.bpart;
            bias.nb[bias.n] = rb;
            bias.out[bias.n] = s->g + c.b_off;
            bias.col[bias.n + 1] = bias.col[bias.n] + c.Cout;
            ++bias.n;
        }
        // weight gradient: dW[co][k] = sum_p g[p][co] col[p][k], the im2col columns gathered by
        // the GEMM's loader when the resolution allows (powers of two), else from a buffer
        GemmArgs gw{};
        gw.conv.x1 = s->t[c.src1].y;
        gw.conv.x2 = c.src2 >= 0 ? s->t[c.src2].y : nullptr;
        gw.conv.C1 = c.C1;
        gw.conv.C2 = c.C2;
        gw.conv.up1 = c.up1;
        gw.conv.H = c.H;
        gw.conv.W = c.W;
        gw.conv.lc = ilog2_exact(Cin);
        gw.conv.lh = ilog2_exact(c.H);
        gw.conv.lw = ilog2_exact(c.W);
        CUtensorMap mx, mdy;
        if (last && conv0_ok(c, gw.conv.x1) && s->splitk_elems >= (size_t)304 * c.Cout * 72 &&
            map_nhwc(&mx, gw.conv.x1, 8, c.W, c.H, B, lbm::sgtc::C0_PITCH, 3, 8) &&
            map_nhwc(&mdy, c.g, c.Cout, c.W, c.H, B, 128, 1, c.Cout)) {
            gw.K = (int)Pc;
            SCUDA(s, c.Cout == 32
                         ? launch_wgrad0<32>(ws, gw, s->splitk, s->g + c.w_off, mx, mdy)
                         : launch_wgrad0<16>(ws, gw, s->splitk, s->g + c.w_off, mx, mdy));
            continue;  // no data gradient for the input tensor
        }
        const bool rows = c.wr_xb != 0, gather = rows || (gw.conv.lh >= 0 && gw.conv.lw >= 0);
        if (!gather && last)  // the side stream's last im2col may still be read
            SCUDA(s, join_side(s));
        if (!gather) SCUDA(s, launch_im2col(s, ws, c, B));
        gw.A = c.g;
        gw.B = s->col;
        gw.M = c.Cout;
        gw.N = 9 * Cin;
        gw.K = (int)Pc;
        gw.lda = c.Cout;
        gw.ldb = 9 * Cin;
        gw.ldc = 9 * Cin;
        float* part = last ? s->splitk : s->splitk_side;
        if (rows) {
            gw.M = 9 * Cin;
            gw.N = c.Cout;
            SCUDA(s, gemm_wgrad_rows(ws, gw, part, s->splitk_elems, s->g + c.w_off, c.wr_xb, c.wr_yb,
                                     c.wr_cb, c.wrmap));
        } else {
            SCUDA(s, gemm_wgrad(ws, gw, part, s->splitk_elems, s->g + c.w_off, gather,
                                gather && c.w_tma ? c.wmap : nullptr));
        }
        // data gradient (not needed for the input tensor)
        if (c.src1 == 0) continue;
        // implicit GEMM over the source pixels: dX_src[q][ci] += sum over (sub-pixel, tap, co)
        // of dY gathered around q times the rearranged weights (no column buffer)
        if (c.up1 && c.C2 > 0) return sfail(s, LBM_ERR_STATE, "surrogate: upsampled cat source");
        GemmArgs gd{};
        gd.dg.dy = c.g;
        gd.dg.H = c.H;
        gd.dg.W = c.W;
        gd.dg.lco = ilog2_exact(c.Cout);
        gd.dg.up1 = c.up1;
        gd.B = s->wbd + c.w_off;
        gd.ldb = 9 * c.Cout;
        gd.kperiod = c.up1 ? 9 * c.Cout : 0;
        gd.M = (int)((long long)B * (c.H >> c.up1) * (c.W >> c.up1));
        gd.N = Cin;
        gd.K = (c.up1 ? 36 : 9) * c.Cout;
        gd.Cf = s->t[c.src1].dy;
        gd.ldc = c.C1;
        if (c.C2 > 0 && written[c.src1] != written[c.src2]) {
            const int fresh = written[c.src1] ? c.src2 : c.src1;
            const Tensor& x = s->t[fresh];
            if (!x.dy) return sfail(s, LBM_ERR_STATE, "surrogate: missing gradient buffer");
            SCUDA(s, cudaMemsetAsync(x.dy, 0, (size_t)B * x.H * x.W * x.C * sizeof(float), s->stream));
            written[fresh] = 1;
        }
        const bool fresh1 = !written[c.src1];
        gd.accumulate = !fresh1;
        written[c.src1] = 1;
        if (c.src2 >= 0) written[c.src2] = 1;
        if (c.C2 > 0) {
            gd.Cf2 = s->t[c.src2].dy;
            gd.ldc2 = c.C2;
            gd.nsplit = c.C1;
        }
        if (c.dm.kb) {
            const Conv* p = fresh1 ? sole_producer(s, c) : nullptr;
            if (p) {
                gd.ry = s->t[c.src1].y;
                gd.rg = p->g;
                gd.rpart = p->bpart;
            }
            SCUDA(s, conv_march<true>(s->stream, gd, c.dm, c.dmmap, &fused[c.src1]));
        } else {
            SCUDA(s, (gemm_tc_split<false, true>(s->stream, gd, s->splitk, s->splitk_elems,
                                                  c.dmap, c.d_ks)));
        }
    }
    SCUDA(s, launch_pdl(k_bias_final, dim3((bias.col[bias.n] + 7) / 8), 256, 0, s->side, bias));
    SCUDA(s, join_side(s));
    if (lr > 0.f) {
        ++s->adam_t;
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.f / (1.f - powf(b1, (float)s->adam_t));
        const float c2 = 1.f / (1.f - powf(b2, (float)s->adam_t));
        SCUDA(s, launch_pdl(k_adam, dim3(s->tab.tile[s->tab.n]), 256, 0, s->stream, s->w, s->g, s->m, s->v,
                            (long long)s->nparams, s->base + 1, lr, b1, b2, 1e-8f, c1, c2, s->wb, s->wbd,
                            s->tab));
    }
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_surrogate_create(int32_t H, int32_t W, int32_t base, int32_t max_batch,
                                int32_t device, lbm_surrogate** out) {
    if (!out) return sfail(nullptr, LBM_ERR_ARG, "lbm_surrogate_create: out is NULL");
    *out = nullptr;
    if (H <= 0 || W <= 0 || H % 8 || W % 8 || (base != 8 && base != 16 && base != 32) ||
        max_batch <= 0)
        return sfail(nullptr, LBM_ERR_ARG,
                     "lbm_surrogate_create: H, W multiples of 8, base 8, 16 or 32, batch > 0");
    if (cudaSetDevice(device) != cudaSuccess) {
        cudaGetLastError();
        return sfail(nullptr, LBM_ERR_CUDA, "lbm_surrogate_create: cannot select the device");
    }
    lbm_surrogate* s = new lbm_surrogate();
    s->H = H;
    s->W = W;
    s->base = base;
    s->maxB = max_batch;
    s->device = device;
    build(s);
    s->tab.n = std::min<int>(24, (int)s->convs.size());  // 17 convolutions
    for (int k = 0; k < s->tab.n; ++k) {
        const Conv& c = s->convs[k];
        s->tab.tile[k + 1] = s->tab.tile[k] + (c.Cout + 31) / 32 * ((9 * (c.C1 + c.C2) + 31) / 32);
        s->tab.off[k] = (long long)s->convs[k].w_off;
        s->tab.cout[k] = s->convs[k].Cout;
        s->tab.cin[k] = s->convs[k].C1 + s->convs[k].C2;
    }
    auto cleanup = [&](const char* e) {
        lbm_surrogate_destroy(s);
        return sfail(nullptr, LBM_ERR_CUDA, std::string("lbm_surrogate_create: ") + e);
    };
    cudaError_t e = cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s->side, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cleanup(cudaGetErrorString(e));
    cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, device);
    const size_t np = s->nparams, px = (size_t)max_batch * H * W;
    size_t wmax = 0;
    for (const Conv& c : s->convs) wmax = std::max(wmax, (size_t)c.Cout * 9 * (c.C1 + c.C2));
    s->splitk_elems = std::min<size_t>(wmax * 128, (size_t)64 << 20);
    std::vector<Part> parts;
    for (size_t k = 1; k < s->t.size(); ++k)
        parts.push_back({(void**)&s->t[k].y, (size_t)max_batch * s->t[k].H * s->t[k].W * s->t[k].C * sizeof(bf16)});
    for (Conv& c : s->convs) {
        parts.push_back({(void**)&c.g, (size_t)max_batch * c.H * c.W * c.Cout * sizeof(bf16)});
        parts.push_back({(void**)&c.bpart, (size_t)kReluBlocks * c.Cout * sizeof(float)});
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c.ready, cudaEventDisableTiming);
    }
    for (float** q : {&s->w, &s->g, &s->m, &s->v}) parts.push_back({(void**)q, np * sizeof(float)});
    for (bf16** q : {&s->wb, &s->wbd}) parts.push_back({(void**)q, np * sizeof(bf16)});
    for (float** q : {&s->dz, &s->phi}) parts.push_back({(void**)q, px * sizeof(float)});
    for (float** q : {&s->splitk, &s->splitk_side}) parts.push_back({(void**)q, s->splitk_elems * sizeof(float)});
    parts.push_back({(void**)&s->hpart, (size_t)s->part_blocks * (base + 2) * sizeof(float)});
    parts.push_back({(void**)&s->n_mask, sizeof(int)});
    if (e == cudaSuccess) e = allocate(s, parts);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->head_ready, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->side_done, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaHostAlloc((void**)&s->host_loss, sizeof(float), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&s->host_loss_dev, s->host_loss, 0);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->w, 0, np * sizeof(float), s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->m, 0, np * sizeof(float), s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->v, 0, np * sizeof(float), s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->wb, 0, np * sizeof(bf16), s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->wbd, 0, np * sizeof(bf16), s->stream);
    if (e != cudaSuccess) return cleanup(cudaGetErrorString(e));
    make_tensor_maps(s);
    // what depends on how the layers run: an im2col buffer for weight gradients that cannot gather, FP32
    // gradients of the activations that a data gradient stores
    std::vector<char> stored(s->t.size(), 1);
    stored[0] = stored[s->head_in] = 0;
    size_t colmax = 0;
    for (const Conv& c : s->convs) {
        if (fused_always(s, c)) stored[c.src1] = 0;
        if (!c.wr_xb && (ilog2_exact(c.H) < 0 || ilog2_exact(c.W) < 0))
            colmax = std::max(colmax, (size_t)max_batch * c.H * c.W * 9 * (c.C1 + c.C2));
    }
    std::vector<size_t> size;  // of the gradient buffers, in values
    const std::vector<int> buf = gradient_buffers(s, stored, &size);
    std::vector<float*> dy(size.size(), nullptr);
    parts.clear();
    for (size_t k = 0; k < size.size(); ++k) parts.push_back({(void**)&dy[k], size[k] * sizeof(float)});
    if (colmax) parts.push_back({(void**)&s->col, colmax * sizeof(bf16)});
    e = allocate(s, parts);
    for (size_t k = 0; k < s->t.size(); ++k)
        if (buf[k] >= 0) s->t[k].dy = dy[buf[k]];
    if (e != cudaSuccess) return cleanup(cudaGetErrorString(e));
    *out = s;
    return LBM_OK;
}

int64_t lbm_surrogate_num_params(const lbm_surrogate* s) { return s ? (int64_t)s->nparams : 0; }

lbm_status lbm_surrogate_set_weights(lbm_surrogate* s, const float* host, int64_t n) {
    if (!s || !host || n != (int64_t)s->nparams)
        return sfail(s, LBM_ERR_ARG, "lbm_surrogate_set_weights: need num_params floats");
    SCUDA(s, cudaSetDevice(s->device));
    SCUDA(s, cudaMemcpyAsync(s->w, host, n * sizeof(float), cudaMemcpyHostToDevice, s->stream));
    SCUDA(s, refresh_bf16_weights(s));
    SCUDA(s, cudaMemsetAsync(s->m, 0, n * sizeof(float), s->stream));
    SCUDA(s, cudaMemsetAsync(s->v, 0, n * sizeof(float), s->stream));
    s->adam_t = 0;
    SCUDA(s, cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

lbm_status lbm_surrogate_get_weights(lbm_surrogate* s, float* host, int64_t n, int32_t grads) {
    if (!s || !host || n != (int64_t)s->nparams)
        return sfail(s, LBM_ERR_ARG, "lbm_surrogate_get_weights: need num_params floats");
    SCUDA(s, cudaSetDevice(s->device));
    SCUDA(s, cudaMemcpyAsync(host, grads ? s->g : s->w, n * sizeof(float), cudaMemcpyDeviceToHost,
                             s->stream));
    SCUDA(s, cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

lbm_status lbm_surrogate_forward(lbm_surrogate* s, const void* x, int32_t B, float* phi_out) {
    lbm::NvtxRange nvtx_("lbm_surrogate_forward");
    if (!s || !x || !phi_out || B <= 0 || B > s->maxB)
        return sfail(s, LBM_ERR_ARG, "lbm_surrogate_forward: bad arguments");
    SCUDA(s, cudaSetDevice(s->device));
    const lbm_status st = settle(s, queue_forward(s, (const bf16*)x, B, phi_out));
    if (st != LBM_OK) return st;
    SCUDA(s, cudaStreamSynchronize(s->stream));
    if (tc_timed_out())
        return sfail(s, LBM_ERR_TIMEOUT, "lbm_surrogate_forward: a tensor-core wait timed out");
    return LBM_OK;
}

// Gradients of the masked MSE into s->g; with lr > 0 also an Adam update. *loss gets the loss.
lbm_status lbm_surrogate_train_step(lbm_surrogate* s, const void* xin, const float* target,
                                    const uint8_t* mask, int32_t B, float lr, double* loss) {
    lbm::NvtxRange nvtx_("lbm_surrogate_train_step");
    if (!s || !xin || !target || !mask || B <= 0 || B > s->maxB)
        return sfail(s, LBM_ERR_ARG, "lbm_surrogate_train_step: bad arguments");
    SCUDA(s, cudaSetDevice(s->device));
    const lbm_status st = settle(s, queue_train_step(s, xin, target, mask, B, lr));
    if (st != LBM_OK) return st;
    SCUDA(s, cudaStreamSynchronize(s->stream));
    if (tc_timed_out())
        return sfail(s, LBM_ERR_TIMEOUT, "lbm_surrogate_train_step: a tensor-core wait timed out");
    if (loss) *loss = *s->host_loss;
    return LBM_OK;
}

lbm_status lbm_surrogate_phi(lbm_surrogate* s, float* host_phi, int32_t B) {
    if (!s || !host_phi || B <= 0 || B > s->maxB)
        return sfail(s, LBM_ERR_ARG, "lbm_surrogate_phi: bad arguments");
    SCUDA(s, cudaMemcpyAsync(host_phi, s->phi, (size_t)B * s->H * s->W * sizeof(float),
                             cudaMemcpyDeviceToHost, s->stream));
    SCUDA(s, cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

// C = A * B with BF16 operands (device), FP32 output; a_kmajor / b_kmajor select the storage
// of A (M x K) and B (K x N): K-major A[m*lda + k], B[n*ldb + k]; MN-major A[k*lda + m],
// B[k*ldb + n].
lbm_status lbm_sg_gemm(const void* A, const void* B, int32_t M, int32_t N, int32_t K,
                       int32_t a_kmajor, int32_t b_kmajor, int32_t lda, int32_t ldb, float* C,
                       int32_t ldc, void* stream) {
    if (!A || !B || !C || M <= 0 || N <= 0 || K <= 0)
        return sfail(nullptr, LBM_ERR_ARG, "lbm_sg_gemm: bad arguments");
    if ((a_kmajor && (K % 8 || lda % 8)) || (!a_kmajor && (M % 8 || lda % 8)) ||
        (b_kmajor && (K % 8 || ldb % 8)) || (!b_kmajor && (N % 8 || ldb % 8)))
        return sfail(nullptr, LBM_ERR_ARG, "lbm_sg_gemm: alignment (multiples of 8) violated");
    if (tc_timed_out())
        return sfail(nullptr, LBM_ERR_TIMEOUT, "lbm_sg_gemm: an earlier tensor-core wait timed out");
    GemmArgs g{};
    g.A = (const bf16*)A;
    g.B = (const bf16*)B;
    g.M = M;
    g.N = N;
    g.K = K;
    g.lda = lda;
    g.ldb = ldb;
    g.Cf = C;
    g.ldc = ldc;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    if (a_kmajor && b_kmajor)
        e = gemm<true, true>(st, g);
    else if (a_kmajor)
        e = gemm<true, false>(st, g);
    else if (b_kmajor)
        e = gemm<false, true>(st, g);
    else
        e = gemm<false, false>(st, g);
    if (e != cudaSuccess)
        return sfail(nullptr, LBM_ERR_CUDA, std::string("lbm_sg_gemm: ") + cudaGetErrorString(e));
    return LBM_OK;
}

// Host-side fault injection: latch the timeout flag exactly as a device wait that ran out
// would, so that callers can exercise their LBM_ERR_TIMEOUT path without stalling a GPU.
lbm_status lbm_sg_inject_timeout(void) {
    TcFlag& f = tc_flag();
    if (!f.host)
        return sfail(nullptr, LBM_ERR_CUDA,
                     "lbm_sg_inject_timeout: the mapped timeout flag could not be allocated");
    *f.host = 1;
    return LBM_OK;
}

void lbm_surrogate_destroy(lbm_surrogate* s) {
    if (!s) return;
    if (s->stream) cudaStreamSynchronize(s->stream);
    if (s->side) cudaStreamSynchronize(s->side);
    for (Conv& c : s->convs)
        if (c.ready) cudaEventDestroy(c.ready);
    if (s->head_ready) cudaEventDestroy(s->head_ready);
    if (s->side_done) cudaEventDestroy(s->side_done);
    for (void* p : s->memory) cudaFree(p);
    if (s->host_loss) cudaFreeHost(s->host_loss);
    if (s->stream) cudaStreamDestroy(s->stream);
    if (s->side) cudaStreamDestroy(s->side);
    delete s;
}

const char* lbm_surrogate_last_error(const lbm_surrogate* s) {
    return s ? s->err.c_str() : lbm_last_error(nullptr);
}

}  // extern "C"

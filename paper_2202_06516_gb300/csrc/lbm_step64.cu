// FP64 time step (Eq. 1-4, 7, 12-14 of arXiv:2202.06516): the step of lbm_step.cu for lattices whose
// populations and densities are doubles, as three kernels.
//
// This chip executes two FP64 lanes per cycle and SM (a warp's FP64 instruction holds the SM's
// FP64 pipe for 16 cycles), so the FP64 step is bound by the number of FP64 operations on every
// lattice size, and by how evenly they are spread over the SMs on small ones; its memory traffic
// (20 planes of 8 bytes per node and step plus 24 of scratch) is far from mattering. The fused
// kernel of the FP32 step recomputes the chemical potential on 1.63 and the collision on 1.2 nodes
// per node of a 32 x 16 tile; here every node's values are computed once and pass through scratch:
//   k64_mu        wetting-layer densities (Eq. 14), then mu (Eq. 12) and the extended density
//   k64_collide   force (Eq. 7), pulled populations (Eq. 4), collision (Eq. 1, 13)
//   k64_stream    rho(t+1) = sum_q f*_q(x - e_q) and the stored deviations
// with 32 or 64 nodes per block, so that a 200 x 120 lattice gives every SM about the same work.
// Only the light k64_stream is placed early (programmatic dependent launch): blocks of the other two
// placed early crowd onto some SMs, and the FP64 pipe of each SM is what the step waits for (44
// against 32 us per step; k64_stream alone placed early: 21.2 to 20.6).
// The operations and their order are those of the fused step; the bulk chemical potential shares one
// reciprocal between its divisions. 200 x 120 (Carnahan-Starling): 64 us per step fused on 56 CTAs,
// 21 us here (k64_mu 8.5, k64_collide 12, k64_stream 5 us each alone and cold).
#include <algorithm>

#include "lbm_step_body.cuh"

namespace lbm {
namespace {

using namespace stepdev;

struct Args64 {
    StepArgs<double> a;
    double rho_mid;
    double c2;            // a alpha / (2 sqrt2 b) of the Peng-Robinson potential
    double *ext, *mu;     // density with wetting layers, chemical potential (rows -2 .. ny + 1)
    double* post;         // 10 planes: post-collision deviations g*_q, and sum_q w_q rho(x - e_q)
};

__device__ __forceinline__ double psi64(double rho, const Args64& s) {
    const StepArgs<double>& a = s.a;
    const double br = a.b * rho;
    if (a.eos == LBM_EOS_PR) {
        // d1 = 1 - b rho, d2 = sqrt2 + 1 - b rho, n2 = sqrt2 - 1 + b rho; 1 + 2 b rho - (b rho)^2 = d2 n2
        const double s2 = 1.4142135623730951;
        const double d1 = 1.0 - br, d2 = (s2 + 1.0) - br, n2 = (s2 - 1.0) + br;
        const double dn = d2 * n2, r = 1.0 / (d1 * dn);
        const double inv_d1 = dn * r, inv_dn = d1 * r;
        return a.RT * (log(rho * inv_d1) + inv_d1) - s.c2 * log(n2 * n2 * inv_dn) -
               a.aal * rho * inv_dn;
    }
    const double n = 0.25 * br, om = 1.0 - n;
    const double num = n * (8.0 + n * (3.0 * n - 9.0));
    return a.RT * (log(rho) + num / (om * om * om)) - 2.0 * a.aal * rho;
}

// 36 / k for the weight sums k / 36 of Eq. 14 (k = 4 per axis neighbour, 1 per diagonal one)
__constant__ double kInvDen[21] = {0.0, 36.0, 18.0, 12.0, 9.0, 36.0 / 5, 6.0, 36.0 / 7, 4.5, 4.0,
                                   3.6, 36.0 / 11, 3.0, 36.0 / 13, 36.0 / 14, 2.4, 2.25, 36.0 / 17,
                                   2.0, 36.0 / 19, 1.8};

// Chemical potential and extended density of an MX x MY block of the rows -2 .. ny + 1. Density
// and classes are staged with four nodes around the block; the first layer is rebuilt on three,
// the second on two nodes around it, as far as the stencil reaches. Three threads per node of the
// block, so that staging and the layers are one or two rounds.
constexpr int MX = 16, MY = 4, MT = 192;
__global__ void __launch_bounds__(MT) k64_mu(const Args64 s) {
    constexpr int W = MX + 8, H = MY + 8, K = (W * H + MT - 1) / MT;
    __shared__ double r[H][W];
    __shared__ uint8_t f[H][W];
    const StepArgs<double>& a = s.a;
    const int x0 = blockIdx.x * MX, y0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * MY - 2;
    const int tid = threadIdx.x;
    int any = 0, e[K];
    uint8_t cl[K];
    double v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int t = tid + k * MT, ly = t / W, lx = t - ly * W, gx = x0 - 4 + lx, gy = y0 - 4 + ly;
        const bool in = ly < H && gx < a.nx + kPadX && gy >= -kPadY && gy < a.ny + kPadY;
        e[k] = in ? lidx(a.P, gx, gy) : -1;
        cl[k] = in ? a.flags[e[k]] : kSolid;
        v[k] = in ? a.rho_in[e[k]] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int t = tid + k * MT, ly = t / W, lx = t - ly * W;
        if (ly >= H) continue;
        f[ly][lx] = cl[k];
        r[ly][lx] = v[k];
        any |= cl[k] != kFluid;
    }
    if (__syncthreads_or(any)) {
        // layer 1 from fluid neighbours, then layer 2 from layer 1 (Eq. 14)
#pragma unroll 1
        for (int layer = 1; layer <= 2; ++layer) {
            const uint8_t match = layer == 1 ? kFluid : kLayer1, mine = layer == 1 ? kLayer1 : kLayer2;
            const int w = W - 2 * layer, h = H - 2 * layer;
            for (int k = tid; k < w * h; k += MT) {
                const int ly = layer + k / w, lx = layer + k % w;
                if (f[ly][lx] != mine) continue;
                double num = 0;
                int den = 0;
#pragma unroll
                for (int q = 1; q < 9; ++q)
                    if (f[ly + qy(q)][lx + qx(q)] == match) {
                        num = fma_rn(qw<double>(q), r[ly + qy(q)][lx + qx(q)], num);
                        den += q <= 4 ? 4 : 1;
                    }
                r[ly][lx] = den > 0 ? num * kInvDen[den] : s.rho_mid;
            }
            __syncthreads();
        }
    }
    if (tid >= MX * MY) return;
    const int tx = tid % MX, ty = tid / MX, gx = x0 + tx, gy = y0 + ty;
    if (gx >= a.nx || gy >= a.ny + 2) return;
    const int ly = ty + 4, lx = tx + 4, at = lidx(a.P, gx, gy);
    const uint8_t c = f[ly][lx];
    const double c0 = r[ly][lx];
    double mu = 0.0;
    if (c == kFluid) {
        const double s1 = add_rn(add_rn(r[ly][lx + 1], r[ly][lx - 1]), add_rn(r[ly + 1][lx], r[ly - 1][lx]));
        const double s2 = add_rn(add_rn(r[ly][lx + 2], r[ly][lx - 2]), add_rn(r[ly + 2][lx], r[ly - 2][lx]));
        const double lap12 = fma_rn(16.0, s1, fma_rn(-60.0, c0, -s2));
        mu = fma_rn(a.k2, psi64(c0, s), mul_rn(mul_rn(a.kappa, -1.0 / 12.0), lap12));
    } else if (c == kLayer1 || c == kLayer2) {
        mu = a.muw[at];
    }
    s.mu[at] = mu;
    s.ext[at] = c0;
}

// x + dx with the periodic images wrapped into 0 .. nx - 1 (|dx| <= 2, nx >= 8)
__device__ __forceinline__ int wrap_x(int x, int nx) { return x < 0 ? x + nx : x >= nx ? x - nx : x; }

constexpr int N64 = 32;  // nodes per block of the two per-node kernels

template <bool MACRO, bool IBB>
__global__ void __launch_bounds__(N64) k64_collide(const Args64 s) {
    const StepArgs<double>& a = s.a;
    pdl_launch_next();
    const int n = blockIdx.x * N64 + threadIdx.x;
    const int y = n / a.nx, x = n - y * a.nx, P = a.P;
    const bool in = y < a.ny;
    const unsigned us = (unsigned)lidx(P, in ? x : 0, in ? y : 0), upl = (unsigned)a.plane;
    // classes of the sources x - e_q; the pads hold the periodic images of flags and populations
    const bool fluid = in && a.flags[us] == kFluid;
    unsigned cut = 0;
    if (fluid)
#pragma unroll
        for (int q = 1; q < 9; ++q)
            if (a.flags[us - qy(q) * P - qx(q)] != kFluid) cut |= 1u << q;
    if (!fluid) return;
    double h[9];
    h[0] = a.h_in[us];
#pragma unroll
    for (int q = 1; q < 9; ++q)
        h[q] = cut >> q & 1 ? a.h_in[(unsigned)qopp(q) * upl + us]
                            : a.h_in[(unsigned)q * upl + us - qy(q) * P - qx(q)];
    int col[5];  // elements of columns x - 2 .. x + 2 in this row (no pads in the scratch planes)
#pragma unroll
    for (int k = -2; k <= 2; ++k) col[k + 2] = lidx(P, wrap_x(x + k, a.nx), y);
    const double* m = s.mu;
    const double* r = s.ext;
    const int c = col[2];
    const double rho = r[c], rE = r[col[3]], rW = r[col[1]], rN = r[c + P], rS = r[c - P];
    const double Gmx = fma_rn(8.0, sub_rn(m[col[3]], m[col[1]]), sub_rn(m[col[0]], m[col[4]]));
    const double Gmy = fma_rn(8.0, sub_rn(m[c + P], m[c - P]), sub_rn(m[c - 2 * P], m[c + 2 * P]));
    const double Grx = fma_rn(8.0, sub_rn(rE, rW), sub_rn(r[col[0]], r[col[4]]));
    const double Gry = fma_rn(8.0, sub_rn(rN, rS), sub_rn(r[c - 2 * P], r[c + 2 * P]));
    const double Fx = fma_rn(rho, fma_rn(Gmx, -1.0 / 12.0, a.gx), fma_rn(Grx, 1.0 / 36.0, a.gbx));
    const double Fy = fma_rn(rho, fma_rn(Gmy, -1.0 / 12.0, a.gy), fma_rn(Gry, 1.0 / 36.0, a.gby));
    // densities of the sources x - e_q
    const double rs[9] = {rho, rW, rS, rE, rN, r[col[1] - P], r[col[3] - P], r[col[3] + P], r[col[1] + P]};
    double g[9], A = mul_rn(qw<double>(0), rho), dm = 0.0;
    g[0] = h[0];
#pragma unroll
    for (int q = 1; q < 9; ++q) {
        if (!(cut >> q & 1)) {
            g[q] = fma_rn(qw<double>(q), sub_rn(rs[q], rho), h[q]);
            A = fma_rn(qw<double>(q), rs[q], A);
            continue;
        }
        g[q] = h[q];
        A = fma_rn(qw<double>(q), rho, A);
        if (IBB) {  // as ibb_return, on the node's neighbour at x + e_q (rs of the opposite direction)
            const double D = a.dlt[(unsigned)(q - 1) * upl + us], D2 = add_rn(D, D);
            if (D >= 0.5) {
                const double ci = recip(D2);
                g[q] = fma_rn(ci, h[q], mul_rn(sub_rn(1.0, ci), a.h_in[(unsigned)q * upl + us]));
            } else if (!(cut >> qopp(q) & 1)) {
                const double hb = a.h_in[(unsigned)qopp(q) * upl + us + qy(q) * P + qx(q)];
                const double behind = fma_rn(qw<double>(q), sub_rn(rs[qopp(q)], rho), hb);
                g[q] = fma_rn(D2, h[q], mul_rn(sub_rn(1.0, D2), behind));
            }
            dm = add_rn(dm, sub_rn(h[q], g[q]));
        }
    }
    if (IBB) g[0] = add_rn(g[0], dm);
    double ux, uy;
    collide<double>(g, rho, Fx, Fy, a, ux, uy);
    if (MACRO) {
        a.vx[us] = ux + 0.5 * Fx / rho;
        a.vy[us] = uy + 0.5 * Fy / rho;
    } else {
#pragma unroll
        for (int q = 0; q < 9; ++q) s.post[(size_t)q * upl + us] = g[q];
        s.post[(size_t)9 * upl + us] = A;
    }
}

__global__ void __launch_bounds__(N64) k64_stream(const Args64 s) {
    const StepArgs<double>& a = s.a;
    const int n = blockIdx.x * N64 + threadIdx.x;
    const int y = n / a.nx, x = n - y * a.nx, P = a.P;
    const bool in = y < a.ny;
    const unsigned us = (unsigned)lidx(P, in ? x : 0, in ? y : 0), upl = (unsigned)a.plane;
    const bool fluid = in && a.flags[us] == kFluid;
    unsigned src[9];
    if (fluid)
#pragma unroll
        for (int q = 1; q < 9; ++q) {
            const bool cut = a.flags[us - qy(q) * P - qx(q)] != kFluid;
            src[q] = cut ? (unsigned)qopp(q) * upl + us
                         : (unsigned)q * upl + (unsigned)lidx(P, wrap_x(x - qx(q), a.nx), y - qy(q));
        }
    pdl_wait_previous();
    if (!fluid) return;
    double g[9], t[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) g[q] = s.post[(size_t)q * upl + us];
#pragma unroll
    for (int q = 1; q < 9; ++q) t[q] = s.post[src[q]];
    const double A = s.post[(size_t)9 * upl + us], r0 = s.ext[us];
    double B = g[0];
#pragma unroll
    for (int q = 1; q < 9; ++q) B = add_rn(B, t[q]);
    const double r1 = add_rn(A, B), dr = sub_rn(r0, r1);
    const bool lo = x < kPadX, hi = x >= a.nx - kPadX;
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        const double v = q < 9 ? fma_rn(qw<double>(q < 9 ? q : 0), dr, g[q < 9 ? q : 0]) : r1;
        double* o = (q < 9 ? a.h_out + (size_t)q * upl : a.rho_out) + us;
        o[0] = v;
        if (lo) o[a.nx] = v;  // periodic images in the pads
        if (hi) o[-a.nx] = v;
    }
}

}  // namespace

size_t step64_scratch_bytes(size_t plane) { return 12 * plane * sizeof(double); }

cudaError_t launch_step64(lbm_ctx* c, const StepArgs<double>& a, bool macro) {
    Args64 s{};
    s.a = a;
    s.rho_mid = 0.5 * (c->rho_g + c->rho_l);
    s.c2 = a.b > 0 ? a.aal / (2.0 * 1.4142135623730951 * a.b) : 0.0;
    s.ext = (double*)c->scratch64;
    s.mu = s.ext + c->plane;
    s.post = s.mu + c->plane;
    // rows of blocks along y and, past the 65535 that y holds (lattices of more than 262136 rows), z
    const unsigned mrows = (c->ny + 4 + MY - 1) / MY, mz = (mrows + 65534) / 65535;
    const dim3 gm((c->nx + MX - 1) / MX, (mrows + mz - 1) / mz, mz);
    const dim3 gn((unsigned)(((long long)c->nx * c->ny + N64 - 1) / N64));
    k64_mu<<<gm, MT, 0, c->stream>>>(s);
    auto* collide = macro ? (c->ibb ? k64_collide<true, true> : k64_collide<true, false>)
                          : (c->ibb ? k64_collide<false, true> : k64_collide<false, false>);
    collide<<<gn, N64, 0, c->stream>>>(s);
    cudaError_t e = cudaGetLastError();
    if (macro || e != cudaSuccess) return e;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = gn;
    cfg.blockDim = dim3(N64);
    cfg.stream = c->stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k64_stream, s);
}

}  // namespace lbm

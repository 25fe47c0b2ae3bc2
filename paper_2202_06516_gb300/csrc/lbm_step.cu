// Fused multiphase LBM time step (Eq. 1-4, 7, 12-14 of arXiv:2202.06516), one launch per step.
//
// Stored state between steps, per fluid node z:
//   rho(z, t)                      density of the current (post-streaming) populations
//   h_q(z) = f*_q(z, t-1) - w_q rho(z, t)
// i.e. the post-collision populations of the previous step as deviations from the rest-state
// equilibrium w_q rho at the node's current density. Deviations are O(rho |u|) and O(f - f_eq),
// so FP32 keeps their relative precision in both phases although the liquid is ~145 times
// denser than the gas; the density itself is stored once per node.
//
// One CTA owns a TX x TY tile and stages, in shared memory:
//   rho, flags   tile + 7    (loaded)
//   wetting layers           first layer on tile + 6, second on tile + 5 (Eq. 14, recomputed
//                            from fluid densities, so no separate boundary kernel runs)
//   mu           tile + 3    (Eq. 12: k^2 psi'(rho) - kappa lap(rho) at fluid nodes, mu_w on the
//                            wetting layers; fourth-order stencils reach 2 nodes)
//   g*           tile + 1    (post-collision deviations from w_q rho(t), collision of Eq. 1 with
//                            force Eq. 7 and exact-difference forcing Eq. 13)
// and writes, for the tile only, rho(t+1) = sum_q f*_q(x - e_q) (pull streaming of Eq. 4 with
// half-way bounce-back on links into the solid) and the new deviations h. Collisions on the
// one-node ring are recomputed by the neighbouring CTAs; that redundancy buys a single pass over
// the populations per step (36 B read + 36 B written + 8 B of density per node in FP32).
#include <algorithm>

#include "lbm_step_body.cuh"

namespace lbm {
namespace {

using namespace stepdev;

// the interpolated bounce-back kernels exist for the default variant (32 x 16 tiles, 5 CTAs per SM)
// and its small-lattice forms; the fractions and populations of a node's cut links in flight take
// registers that five CTAs per SM would spill. us per step with a cylinder: five CTAs and a chain of two
// latencies per cut link / four / five that spill 56 bytes: 640x480 19.5 / 16.0 / 16.2, 768x480 20.1 / 16.2 /
// 18.4, 1024x512 22.3 / 17.9 / 18.9, 1500x701 32.0 / 28.5 / 27.6, 2048x1024 55.7 / 51.6 / 48.5
constexpr int kIbbBlocks = 4;
template <typename T, int TX, int TY, int MINB>
constexpr bool has_ibb() {
    return TX == 32 && TY == 16 && MINB == 5;
}

// Launch with programmatic stream serialization (early): a step's launch, block placement and class
// staging overlap the previous step's tail (k_step waits before it reads what that step wrote).
template <typename T, int TX, int TY, int NT, int MINB, bool MACRO, bool IBB>
cudaError_t launch_k(lbm_ctx* c, const StepArgs<T>& a, bool early) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((c->nx + TX - 1) / TX, (c->ny + TY - 1) / TY);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = Layout<T, TX, TY>::bytes;
    cfg.stream = c->stream;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_step<T, TX, TY, NT, MACRO, MINB, IBB>, a,
                              (T)(0.5 * (c->rho_g + c->rho_l)));
}

template <typename T, int TX, int TY, int NT, int MINB, bool MACRO, bool IBB>
cudaError_t allow_smem() {
    return cudaFuncSetAttribute(k_step<T, TX, TY, NT, MACRO, MINB, IBB>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Layout<T, TX, TY>::bytes);
}

// Small-lattice forms of the default FP32 variant. A step of a small lattice is one chain of
// latencies (launch, staging, wetting layers, chemical potential, gathers, streaming, each with its
// barrier) on a chip that is mostly idle, so these forms give a tile so many threads that
// every stage is one round, or spread the lattice over more, smaller tiles; on large lattices the
// recomputed halo and the fewer resident tiles make them slower. Chosen by the number of tiles
// against the number of SMs. They are for one lattice at a time: with the chip full of lattices on streams of
// their own the recomputed halos count (16 of 200x120 at once 12.5 us per step of all with 256 threads, 18.0
// with form 1; 256x256 23.6, 53.6; 520x190 36.8, 56.5), which a lattice cannot know: 32x16/5 by name leaves them out.
// Measured, us per step, 32x16 tiles of 256 threads / forms 1 / 2 / 3:
// 128x96 7.4 / 4.3 / 5.1 / 4.8; 200x120 8.0 / 4.6 / 5.1 / 5.2; 256x256 8.0 / 6.0 / 5.2 / 5.6;
// 520x190 10.2 / 6.8 / 7.2 / 6.1.
// Form 3 holds three tiles per SM (456); up to twice as many run as a second wave. It then pays, the more
// where a curved wall crosses tiles (the 256-thread form's threads take several rounds of wetting layers
// and cut links there), until the second wave is nearly full; half-way walls, us per step, 256 threads /
// form 3: flat 700x165 (462 tiles) 8.2 / 6.6, 400x324 (533) 7.4 / 7.3, 700x216 (594) 9.0 / 7.6, 400x397
// (650) 9.0 / 8.1, 1100x160 (700) 9.2 / 8.3, 700x278 (770) 9.3 / 8.7, 250x835 (840) 9.5 / 9.4, 1100x192 (840) 9.0 /
// 9.2, 1100x200 (875) 8.5 / 9.5, 400x548 (897) 9.2 / 9.5; R = 24 within 0.2 of flat; R = 48 250x835 9.7 / 9.4,
// 1100x200 9.9 / 9.6. Where the 256-thread form needs a fourth tile per SM: 700x322 (902) 11.0 / 9.7.
// Lattices of up to four columns of tiles have few wall tiles but many that write pads, which costs form 3
// more, and R decides: flat 128x956 (480) 7.0 / 6.9, 128x1197 (600) 7.0 / 7.5, 128x1316 (660) 8.7 / 7.8,
// 128x1440 (720) 8.6 / 8.0, 128x1560 (780) 7.7 / 8.9, 40x2399 (600) 7.3 / 8.2, 40x2635 (660) 8.7 / 8.8, 40x3119 (780) 8.7 /
// 9.5 (beyond two tiles of 32x16 per SM, at about 608 of 32x8, the 256-thread form steps up); R = 24 128x1197
// 8.1 / 7.5, 128x1440 8.9 / 8.1, 128x1806 (904) 8.9 / 9.2; R = 48 128x1560 10.2 / 8.9, 128x1806 10.2 / 9.3. A cavity
// leaves most tiles empty: 700x328 (902) 11.4 / 10.3, 1000x224 (896) 11.3 / 9.1. Interpolated walls take longer in
// the 256-thread form at every size: 128x1200 (600), R = 3, 10.5 / 9.2, 512x456 (912) 15.0 / 11.1.
#define LBM_SMALL_FORMS(X) X(1, 16, 8, 320, 3) X(2, 32, 16, 640, 1) X(3, 32, 8, 384, 3)

// tiles of tx x ty nodes that hold a fluid node (c->geom); the others leave after staging
long long fluid_tiles(const lbm_ctx* c, int tx, int ty) {
    const long long cols = (c->nx + tx - 1) / tx, rows = (c->ny + ty - 1) / ty;
    const lbm_geometry& g = c->geom;
    if (!g.has_circle) return cols * rows;
    long long n = 0;
    for (long long r = 0; r < rows; ++r) {
        const double y0 = (double)(r * ty), y1 = std::min<double>(y0 + ty, c->ny) - 1;
        // rows of the tile against the circle: the nearest one (cavity) or the farthest one (cylinder)
        const double dy = g.concave ? std::max({0.0, y0 - g.cy, g.cy - y1})
                                    : std::max(fabs(y0 - g.cy), fabs(y1 - g.cy));
        const double h2 = g.R * g.R - dy * dy;
        const double lo = h2 >= 0 ? g.cx - sqrt(h2) : 1, hi = h2 >= 0 ? g.cx + sqrt(h2) : 0;
        if (g.concave) {  // tiles that reach into the cavity
            const double a = std::max(lo, 0.0), b = std::min(hi, c->nx - 1.0);
            if (a <= b) n += (long long)(b / tx) - (long long)(a / tx) + 1;
        } else {  // tiles that do not lie inside the cylinder
            const double a = std::max(ceil(lo / tx), 0.0);
            const double b = hi >= c->nx - 1 ? cols - 1.0 : floor((hi + 1) / tx) - 1;
            n += cols - (lo <= hi && a <= b ? (long long)(b - a) + 1 : 0);
        }
    }
    return n;
}

// Whether a step of the 256-thread forms is placed early. A grid that fits on the chip at once leaves
// slots free, and early placement fills those as they are: some SMs get five tiles of the next step,
// others two, and the step waits for the fullest SM. Placed after the previous step the tiles are
// spread evenly. us per step, half-way walls, drop on a cylinder / in a cavity, early -> not:
// 517x425 (459 tiles) 11.8 -> 10.0 / 13.5 -> 11.0; 640x480 (600) 11.9 -> 11.3 / 13.6 -> 12.8; 768x480
// (720) 12.5 -> 12.3 / 14.0 -> 14.4. Larger grids gain from early placement: 1024x512 (1024 tiles)
// not 16.2, early 15.6 / 16.5, 16.3; 2048x1024 (4096) 46.4, 45.8. Tiles without fluid nodes leave at once, so a
// grid that does not fit behaves like one that does when few of its tiles hold fluid. Cavities, fluid
// tiles / early -> not: 1892x200 271 10.5 -> 9.4; 502x825 405 13.0 -> 10.5; 560x1100 499 13.2 -> 12.2; 620x660 606 13.5 ->
// 13.1; 640x1000 648 13.7 -> 13.6; 1300x380 660 13.5 -> 13.9; 800x560 753 14.0 -> 14.4. Cylinders, whose empty tiles come
// first: 900x440 365 11.7 -> 10.9, 768x512 432 12.0 -> 10.8, 800x520 460 11.5 -> 12.0, 640x620 551 11.3 -> 11.7.
bool launch_early(const lbm_ctx* c) {
    const int tx = c->tile_x, ty = c->tile_y;
    const long long grid = (long long)((c->nx + tx - 1) / tx) * ((c->ny + ty - 1) / ty);
    return grid > c->resident[c->ibb ? 1 : 0] &&
           fluid_tiles(c, tx, ty) > (c->geom.concave ? 4 : 3) * c->sms;
}

// CTAs of a kernel that the whole chip holds at once
template <typename K>
cudaError_t resident_ctas(const lbm_ctx* c, K* kernel, int threads, size_t smem, int* out) {
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    *out = per_sm * c->sms;
    return e;
}

template <typename T, int TX, int TY, int MINB>
cudaError_t configure_one(lbm_ctx* c) {
    cudaError_t e = allow_smem<T, TX, TY, 256, MINB, false, false>();
    if (e == cudaSuccess) e = allow_smem<T, TX, TY, 256, MINB, true, false>();
    if (e == cudaSuccess)
        e = resident_ctas(c, k_step<T, TX, TY, 256, false, MINB, false>, 256, Layout<T, TX, TY>::bytes,
                          &c->resident[0]);
    if constexpr (has_ibb<T, TX, TY, MINB>()) {
        if (e == cudaSuccess) e = allow_smem<T, TX, TY, 256, kIbbBlocks, false, true>();
        if (e == cudaSuccess) e = allow_smem<T, TX, TY, 256, kIbbBlocks, true, true>();
        if (e == cudaSuccess)
            e = resident_ctas(c, k_step<T, TX, TY, 256, false, kIbbBlocks, true>, 256,
                              Layout<T, TX, TY>::bytes, &c->resident[1]);
    }
    if constexpr (has_ibb<T, TX, TY, MINB>()) {
#define X(F, A, B, N, M)                                                       \
    if (e == cudaSuccess) e = allow_smem<float, A, B, N, M, false, false>();   \
    if (e == cudaSuccess) e = allow_smem<float, A, B, N, M, false, true>();
        LBM_SMALL_FORMS(X)
#undef X
    }
    return e;
}

template <typename T, int TX, int TY, int MINB>
cudaError_t launch_one(lbm_ctx* c, const StepArgs<T>& a, bool macro) {
    if constexpr (has_ibb<T, TX, TY, MINB>()) {
        const int form = macro ? 0 : c->form;
#define X(F, A, B, N, M)                                                       \
    if (form == F)                                                             \
        return c->ibb ? launch_k<float, A, B, N, M, false, true>(c, a, true)   \
                      : launch_k<float, A, B, N, M, false, false>(c, a, true);
        LBM_SMALL_FORMS(X)
#undef X
    }
    const bool early = c->early;
    if (c->ibb) {
        if constexpr (has_ibb<T, TX, TY, MINB>())
            return macro ? launch_k<T, TX, TY, 256, kIbbBlocks, true, true>(c, a, early)
                         : launch_k<T, TX, TY, 256, kIbbBlocks, false, true>(c, a, early);
        return cudaErrorInvalidValue;
    }
    return macro ? launch_k<T, TX, TY, 256, MINB, true, false>(c, a, early)
                 : launch_k<T, TX, TY, 256, MINB, false, false>(c, a, early);
}

template <typename T>
StepArgs<T> make_args(lbm_ctx* c, int src) {
    StepArgs<T> a{};
    a.h_in = (const T*)c->h[src];
    a.h_out = (T*)c->h[src ^ 1];
    for (int q = 0; q < 9; ++q) {
        a.hq_in[q] = a.h_in + (size_t)q * c->plane;
        a.hq_out[q] = a.h_out + (size_t)q * c->plane;
    }
    a.rho_in = (const T*)c->rho[src];
    a.rho_out = (T*)c->rho[src ^ 1];
    a.flags = c->flags;
    a.muw = (const T*)c->muw;
    a.dlt = (const T*)c->dlt;
    a.vx = (T*)c->vel;
    a.vy = c->vel ? (T*)c->vel + c->plane : nullptr;
    a.nx = c->nx;
    a.ny = c->ny;
    a.P = c->P;
    a.plane = (int)c->plane;
    a.k2 = (T)c->p.k2;
    a.kappa = (T)c->p.kappa;
    a.gx = (T)c->p.gx;
    a.gy = (T)c->p.gy;
    a.gbx = (T)(-c->p.g_rho_ref * c->p.gx);
    a.gby = (T)(-c->p.g_rho_ref * c->p.gy);
    a.s_e = (T)c->p.s_e;
    a.s_eps = (T)c->p.s_eps;
    a.s_q = (T)c->p.s_q;
    a.s_v = (T)(1.0 / c->p.tau);
    a.inv_tau = (T)(1.0 / c->p.tau);
    a.bgk = c->p.collision == LBM_BGK;
    a.eos = c->eosc.eos;
    a.RT = (T)c->eosc.RT;
    a.aal = (T)c->eosc.aal;
    a.b = (T)c->eosc.b;
    return a;
}

}  // namespace

// Supported step-kernel variants: tile (TX, TY) and the minimum resident CTAs per SM the
// compiler is asked to fit (register budget); min_blocks 0 = no constraint. FP64 lattices step
// with the kernels of lbm_step64.cu, which have no tiles: both names select them.
#define LBM_STEP_VARIANTS(X)                                     \
    X(float, 32, 8, 1) X(float, 32, 8, 6) X(float, 32, 16, 1)    \
    X(float, 32, 16, 5) X(float, 32, 16, 6) X(float, 64, 16, 1)  \
    X(float, 32, 32, 1) X(double, 32, 8, 1) X(double, 32, 16, 1)

static int minb_of(lbm_ctx* c) { return c->min_blocks > 0 ? c->min_blocks : 1; }

size_t step_smem_bytes(int tx, int ty, size_t esz, int min_blocks) {
    const int mb = min_blocks > 0 ? min_blocks : 1;
#define X(T, A, B, M) \
    if (esz == sizeof(T) && tx == A && ty == B && mb == M) return Layout<T, A, B>::bytes;
    LBM_STEP_VARIANTS(X)
#undef X
    return 0;
}

bool step_has_ibb(size_t esz, int tx, int ty, int min_blocks) {
    return tx == 32 && ty == 16 && min_blocks == (esz == 4 ? 5 : 0);
}

void step_variants(size_t esz, std::vector<StepVariant>* out) {
    out->clear();
#define X(T, A, B, M) \
    if (esz == sizeof(T)) out->push_back(StepVariant{A, B, M == 1 ? 0 : M});
    LBM_STEP_VARIANTS(X)
#undef X
}

static int step_form(const lbm_ctx* c) {
    if (c->fixed) return 0;
    const long long nx = c->nx, ny = c->ny, sms = c->sms;
    auto tiles = [&](long long tx, long long ty) {
        return ((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
    };
    if (2 * tiles(16, 8) <= 3 * sms) return 1;
    if (tiles(32, 16) <= sms) return 2;
    const lbm_geometry& g = c->geom;
    const double R = g.has_circle ? g.R : 0;
    const long long large = tiles(32, 16);
    const int quarters = c->ibb || (g.has_circle && g.concave) ? 24  // tiles of 32x8 per SM, times four
                         : nx <= 4 * 32 ? (R >= 32 ? 24 : R >= 16 ? 20 : large > 2 * sms ? 19 : 15)
                         : large > 3 * sms ? 24
                                           : (R >= 32 ? 23 : 22);
    return 4 * tiles(32, 8) <= quarters * sms ? 3 : 0;
}

bool step_choose(lbm_ctx* c) {
    const int form = step_form(c);
    const bool early = launch_early(c), changed = form != c->form || early != c->early;
    c->form = form;
    c->early = early;
    return changed;
}

cudaError_t step_configure(lbm_ctx* c) {
    cudaError_t e = cudaErrorInvalidValue;
#define X(T, A, B, M)                                                                       \
    if (c->esz == sizeof(T) && c->tile_x == A && c->tile_y == B && minb_of(c) == M) {       \
        e = cudaSuccess;                                                                    \
        if constexpr (sizeof(T) == 4) e = configure_one<T, A, B, M>(c);                      \
    }
    LBM_STEP_VARIANTS(X)
#undef X
    step_choose(c);
    return e;
}

cudaError_t launch_step(lbm_ctx* c, int src, bool macro) {
    if (c->esz == 8) return launch_step64(c, make_args<double>(c, src), macro);
    const StepArgs<float> a = make_args<float>(c, src);
#define X(T, A, B, M)                                                                 \
    if constexpr (sizeof(T) == 4)                                                     \
        if (c->tile_x == A && c->tile_y == B && minb_of(c) == M)                      \
            return launch_one<float, A, B, M>(c, a, macro);
    LBM_STEP_VARIANTS(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace lbm

// Reductions and the on-device contact-angle measurement (Sec. 3.2, Eq. 15, Fig. 1-2).
//
// Reductions (mass, liquid-node count and centroid): one kernel, deterministic. Every block writes
// its partial sums to scratch, and the block that finishes last adds them in a fixed order.
//
// Measurement: the threads scan the nodes near the wall surface (a list made with the geometry)
// for liquid/gas links (one end rho > rho_m, the other not) in the four undirected link directions, place the Eq. 15 point on the link, measure its
// distance d to the substrate and keep, per side, the links nearest to d = 1 and d = 2 within
// the band 0.5 <= d <= 2.5 (ordered by |d - target|, then link id). Blocks reduce with warp
// shuffles into per-block partials; the last block to finish picks the winners and builds the
// line, the contact point and the angle. The point and distance arithmetic uses explicitly
// rounded FP64 operations (no contraction), so the candidate set and the chosen links are
// reproducible bit for bit by any IEEE implementation that evaluates the same operations.
//
// Both kernels write their results straight into mapped host memory, so a call is one or two
// launches and one stream synchronisation.
#include <math.h>

#include "lbm_internal.cuh"
#include "lbm_sum.cuh"

namespace lbm {
namespace {

struct Best {
    double key;
    long long id;
    double px, py, d;
};

// keys are non-negative, so their order is that of their bit patterns (integer comparisons: the FP64
// pipe takes two lanes per cycle and SM)
__device__ __forceinline__ bool better(double k1, long long i1, double k2, long long i2) {
    const long long a = __double_as_longlong(k1), b = __double_as_longlong(k2);
    return a < b || (a == b && i1 < i2);
}

__device__ __forceinline__ void shfl_best(Best& b, int o) {
    Best c;
    c.key = __shfl_down_sync(0xffffffffu, b.key, o);
    c.id = __shfl_down_sync(0xffffffffu, b.id, o);
    c.px = __shfl_down_sync(0xffffffffu, b.px, o);
    c.py = __shfl_down_sync(0xffffffffu, b.py, o);
    c.d = __shfl_down_sync(0xffffffffu, b.d, o);
    if (better(c.key, c.id, b.key, b.id)) b = c;
}

// link slots: the four undirected D2Q9 link directions (1,0), (0,1), (1,1), (-1,1)
__device__ __forceinline__ int slot_x(int sl) { return sl == 1 ? 0 : (sl == 3 ? -1 : 1); }
__device__ __forceinline__ int slot_y(int sl) { return sl == 0 ? 0 : 1; }

// Sums of one block, one plane per quantity: mass[nb], then n_liquid, sx, sy, bad [nb] as integers.
struct Partials {
    double* mass;
    unsigned long long* cnt;  // 4 planes
};

// one node's density into the sums; a density that is not a positive finite number is counted
__device__ __forceinline__ void add_node(FixSum& m, unsigned& nbad, float v) {
    if (fix_ok(v)) {
        m.add(to_fix(v));
    } else {
        m.acc += (double)v;
        if (!(v > 0.f) || !isfinite(v)) ++nbad;
    }
}
__device__ __forceinline__ void add_node(FixSum& m, unsigned& nbad, double v) {
    m.acc += v;
    if (!(v > 0.0) || !isfinite(v)) ++nbad;
}

// Mass, liquid count, liquid centroid and the count of non-finite or non-positive densities over
// the fluid nodes, eight nodes per thread and access, 2^lt threads per row: one block per row (then
// striding), or several rows at once where a lattice has more rows than blocks and rows that need few
// threads (8 x 100000, host to host: 84 us with one row per block, 22 so). Bound by
// the 5 bytes per node it reads and, with few rows, by latency: a block's mass is summed in exact
// fixed point (lbm_sum.cuh) and the blocks' in FP64, counts and coordinate sums are integers (the same values the FP64
// sums of whole numbers had), and the comparison with rho_m is made against the largest T not
// above it (the same truth value for every T), so that FP32 lattices use the FP64 pipe only
// for the blocks' totals. 4096 x 1024: 82 us and 26 us for a serial last pass
// (every operation in FP64) became 20 us; 200 x 120: 7 + 26 us became 8.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    k_reduce(const T* rho, const uint8_t* flags, int nx, int ny, int P, int lt, T thr, Partials part,
             unsigned* ticket, ReduceOut* out, ReduceOut* host_out) {
    FixSum mass;
    unsigned long long cnt[4] = {0, 0, 0, 0};  // n_liquid, sx, sy, bad
    const int groups = (nx + 7) / 8;
    const int rows = kRedThreads >> lt;
    for (int j = blockIdx.x * rows + (threadIdx.x >> lt); j < ny; j += gridDim.x * rows) {
        const int row = lidx(P, 0, j);
        unsigned nl = 0, nbad = 0;
        unsigned long long sx = 0;
        for (int g = threadIdx.x & ((1 << lt) - 1); g < groups; g += 1 << lt) {
            const int i0 = 8 * g;
            T v[8];
            load8(rho + row + i0, v);  // columns past nx lie in the row's pad
            const uint2 f = __ldg(reinterpret_cast<const uint2*>(flags + row + i0));
            mass.make_room(8);
            unsigned top = 0;  // FP32: the largest fix_key of the eight
            if constexpr (sizeof(T) == 4) {
#pragma unroll
                for (int k = 0; k < 8; ++k) top = max(top, fix_key(v[k]));
            }
            if (sizeof(T) == 4 && (f.x | f.y) == 0 && i0 + 8 <= nx && top < kFixRange) {
                // eight ordinary fluid nodes
                if constexpr (sizeof(T) == 4) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) mass.add(to_fix(v[k]));
                    if (__uint_as_float(top + kFixLo) > thr) {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (v[k] > thr) {
                                ++nl;
                                sx += (unsigned)(i0 + k);
                            }
                    }
                }
                continue;
            }
#pragma unroll 1
            for (int k = 0; k < 8; ++k) {
                const unsigned fk = ((k < 4 ? f.x : f.y) >> (8 * (k & 3))) & 0xFFu;
                if (fk != kFluid || i0 + k >= nx) continue;
                T x = v[0];
#pragma unroll
                for (int m = 1; m < 8; ++m) x = k == m ? v[m] : x;
                add_node(mass, nbad, x);
                if (x > thr) {
                    ++nl;
                    sx += (unsigned)(i0 + k);
                }
            }
        }
        cnt[0] += nl;
        cnt[1] += sx;
        cnt[2] += (unsigned long long)nl * (unsigned)j;
        cnt[3] += nbad;
    }
    __shared__ double s_acc[kRedThreads / 32];
    __shared__ long long s_fix[kRedThreads / 32];
    __shared__ unsigned long long s_cnt[4][kRedThreads / 32];
    __shared__ int s_last;
    const int nb = gridDim.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a block without liquid or bad nodes (most of them) has four zero counts
    const int has_cnt = __syncthreads_or(cnt[0] != 0 || cnt[3] != 0);
    if (has_cnt)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long u = warp_sum(cnt[k]);
            if (lane == 0) s_cnt[k][warp] = u;
        }
    const double m = block_sum(mass, s_fix, s_acc);
    if (threadIdx.x == 0) part.mass[blockIdx.x] = m;
    if (threadIdx.x < 4) {
        unsigned long long u = 0;
        if (has_cnt)
            for (int w = 0; w < kRedThreads / 32; ++w) u += s_cnt[threadIdx.x][w];
        part.cnt[(size_t)threadIdx.x * nb + blockIdx.x] = u;
    }
    if (!last_block(ticket, gridDim.x, &s_last)) return;
    double md = 0;
    unsigned long long c[4] = {0, 0, 0, 0};
    for (int b = threadIdx.x; b < nb; b += kRedThreads) {
        md += __ldcg(part.mass + b);
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] += __ldcg(part.cnt + (size_t)k * nb + b);
    }
    md = warp_sum(md);
    if (lane == 0) s_acc[warp] = md;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned long long u = warp_sum(c[k]);
        if (lane == 0) s_cnt[k][warp] = u;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        md = 0;
        for (int w = 0; w < kRedThreads / 32; ++w) md += s_acc[w];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c[k] = 0;
            for (int w = 0; w < kRedThreads / 32; ++w) c[k] += s_cnt[k][w];
        }
        ReduceOut r{};
        const double n = (double)c[0];
        r.mass = md;
        r.n_liquid = n;
        r.sx = c[0] ? (double)c[1] / n : 0.0;
        r.sy = c[0] ? (double)c[2] / n : 0.0;
        r.bad = (double)c[3];
        *out = r;
        if (host_out) *host_out = r;
    }
}

// Eq. 15 point of the link from node (i, j) with density va along slot sl to a fluid node with
// density vb, if it joins liquid and gas. thr: the largest T not above rho_m (rho > rho_m exactly
// when rho > thr).
template <typename T>
__device__ __forceinline__ bool link_point(T va, T vb, double rho_m, T thr, int i, int j, int sl,
                                           double& px, double& py) {
    const bool la = va > thr, lb = vb > thr;
    if (la == lb) return false;
    const double ra = (double)va, rb = (double)vb;
    const int ti = i + slot_x(sl), tj = j + slot_y(sl);
    double xg, yg, rg, rl, ex, ey;
    if (la) {
        xg = ti; yg = tj; rg = rb; rl = ra; ex = -slot_x(sl); ey = -slot_y(sl);
    } else {
        xg = i; yg = j; rg = ra; rl = rb; ex = slot_x(sl); ey = slot_y(sl);
    }
    const double fr = __ddiv_rn(__dsub_rn(rho_m, rg), __dsub_rn(rl, rg));
    px = __dadd_rn(xg, __dmul_rn(fr, ex));
    py = __dadd_rn(yg, __dmul_rn(fr, ey));
    return true;
}

// Densities at the other ends of node (i, j)'s four links; bit sl of the result: that end exists
// and is fluid
template <typename T>
__device__ __forceinline__ unsigned link_ends(const T* rho, const uint8_t* flags, int nx, int ny,
                                              int P, int i, int j, T (&vb)[4]) {
    unsigned ok = 0;
#pragma unroll
    for (int sl = 0; sl < 4; ++sl) {
        const int ti = i + slot_x(sl), tj = j + slot_y(sl);
        const int wi = ti < 0 ? ti + nx : (ti >= nx ? ti - nx : ti);
        const int e = lidx(P, wi, tj);  // row ny is a pad row of the planes
        vb[sl] = rho[e];
        if (tj < ny && flags[e] == kFluid) ok |= 1u << sl;
    }
    return ok;
}

// distance from the wall surface into the fluid
__device__ __forceinline__ double substrate_dist(const Substrate& s, double px, double py) {
    if (s.circle) {
        const double dx = __dsub_rn(px, s.cx), dy = __dsub_rn(py, s.cy);
        const double r = __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
        return s.concave ? __dsub_rn(s.Rs, r) : __dsub_rn(r, s.Rs);
    }
    return __dsub_rn(py, -0.5);
}

// Bit sl: the link of fluid node (i, j) along slot sl joins liquid and gas and its point may lie in
// the measurement's band. PRE: points whose FP32 distance is more than a quarter outside the band
// are dropped here. Coordinates and radii up to 10^6 make that distance err by less than 0.2; the
// point's share of the link errs by up to 4 x 2^-24 rho_m / |vb - va| (the roundings of rho_m and of
// both ends), so links whose ends differ by less than 1e-4 rho_m stay in, and for the others that is
// below 0.0025 (0.0036 of distance).
template <typename T, bool PRE>
__device__ __forceinline__ unsigned crossing_links(T va, const T (&vb)[4], unsigned ends, double rho_m,
                                                   T thr, const Substrate& sub, int i, int j) {
    unsigned m = 0;
#pragma unroll
    for (int sl = 0; sl < 4; ++sl) {
        if (!(ends >> sl & 1) || (va > thr) == (vb[sl] > thr)) continue;
        if (PRE) {
            const float a = (float)va, w = (float)vb[sl] - a;
            const bool apart = fabsf(w) >= 1e-4f * (float)rho_m;
            const float fr = __fdividef((float)rho_m - a, w);
            const float x = i + fr * slot_x(sl), y = j + fr * slot_y(sl);
            float d = y + 0.5f;
            if (sub.circle) {
                const float dx = x - (float)sub.cx, dy = y - (float)sub.cy;
                d = sqrtf(dx * dx + dy * dy) - (float)sub.Rs;
                if (sub.concave) d = -d;
            }
            if (apart && (d < 0.25f || d > 2.75f)) continue;
        }
        m |= 1u << sl;
    }
    return m;
}

// The link's point, if in the band, into the four running bests (side * 2 + target)
template <typename T>
__device__ __forceinline__ bool take_link(long long id, int nx, T va, T vb, double rho_m, T thr,
                                          const Substrate& sub, double qxc, double qyc, Best (&b)[4]) {
    const long long n = id >> 2;
    const int sl = (int)(id & 3), j = (int)(n / nx), i = (int)(n - (long long)j * nx);
    double px, py;
    if (!link_point<T>(va, vb, rho_m, thr, i, j, sl, px, py)) return false;
    const double d = substrate_dist(sub, px, py);
    if (!(d >= 0.5 && d <= 2.5)) return false;
    int side;
    if (sub.circle) {
        const double ax = __dsub_rn(qxc, sub.cx), ay = __dsub_rn(qyc, sub.cy);
        const double bx = __dsub_rn(px, sub.cx), by = __dsub_rn(py, sub.cy);
        const double cr = __dsub_rn(__dmul_rn(ax, by), __dmul_rn(ay, bx));
        // the wall normal into the fluid at the centroid is (ax, ay) on the convex
        // circle and -(ax, ay) on the concave one
        side = (sub.concave ? cr < 0.0 : cr > 0.0) ? 0 : 1;
    } else {
        side = px < qxc ? 0 : 1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if ((k >> 1) != side) continue;
        const double key = fabs(__dsub_rn(d, (double)((k & 1) + 1)));
        if (better(key, id, b[k].key, b[k].id)) b[k] = Best{key, id, px, py, d};
    }
    return true;
}

// The line of one side through its two points, its contact point and the wall tangent toward the
// liquid (Fig. 1, Fig. 2); false (and the status set) where the side has none.
__device__ bool side_line(const Best& b1, const Best& b2, const Substrate& sub, int side,
                          lbm_angle* o, double& ct, double& at) {
    o->status = LBM_OK;
    if (!(b1.key < INFINITY) || !(b2.key < INFINITY) || b1.id == b2.id) {
        o->status = LBM_ERR_NO_CONTACT;
        return false;
    }
    o->p1_x = b1.px; o->p1_y = b1.py; o->d1 = b1.d; o->link1 = b1.id;
    o->p2_x = b2.px; o->p2_y = b2.py; o->d2 = b2.d; o->link2 = b2.id;
    double vx = b2.px - b1.px, vy = b2.py - b1.py;
    const double vl = sqrt(vx * vx + vy * vy);
    vx /= vl;
    vy /= vl;
    double Cx, Cy, tx, ty;
    if (sub.circle) {
        const double wx = b1.px - sub.cx, wy = b1.py - sub.cy;
        const double wv = wx * vx + wy * vy;
        const double disc = wv * wv - (wx * wx + wy * wy - sub.Rs * sub.Rs);
        if (disc < 0) {
            o->status = LBM_ERR_NO_CONTACT;
            return false;
        }
        const double sq = sqrt(disc);
        const double s1 = -wv - sq, s2 = -wv + sq;
        const double sc = fabs(s1) < fabs(s2) ? s1 : s2;
        Cx = b1.px + sc * vx;
        Cy = b1.py + sc * vy;
        double nxr = Cx - sub.cx, nyr = Cy - sub.cy;
        const double nl = sqrt(nxr * nxr + nyr * nyr);
        nxr /= nl;
        nyr /= nl;
        if (sub.concave) {  // wall normal into the fluid points to the centre
            nxr = -nxr;
            nyr = -nyr;
        }
        // tangent toward the liquid: clockwise on the left side, counter-clockwise on the right
        if (side == 0) {
            tx = nyr;
            ty = -nxr;
        } else {
            tx = -nyr;
            ty = nxr;
        }
    } else {
        if (vy == 0) {
            o->status = LBM_ERR_NO_CONTACT;
            return false;
        }
        const double sc = (-0.5 - b1.py) / vy;
        Cx = b1.px + sc * vx;
        Cy = -0.5;
        tx = side == 0 ? 1.0 : -1.0;
        ty = 0.0;
    }
    ct = fmin(1.0, fmax(-1.0, tx * vx + ty * vy));
    at = fmin(1.0, fabs(tx));
    o->contact_x = Cx;
    o->contact_y = Cy;
    return true;
}

// Both contact angles. The nodes scanned are the listed ones (a few thousand on the wall, against
// millions in the lattice: the whole-lattice scan it replaces took 152 us on 4096 x 1024 and 18 us on
// 200 x 120) or, where the list could not be made (band_n negative or above cap), every fluid
// node. The order of the list does not matter: the winners are minima by (key, link id). Chains of
// dependent FP64 operations are what this kernel costs, so a block first collects its crossing
// links (FP32 work) and then gives each thread one of them, and the block that finishes last
// builds the angles with one warp per (side, angle). Four links in turn per thread took 25 us.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    k_measure(const T* rho, const uint8_t* flags, int nx, int ny, int P, double rho_m, T thr,
              Substrate sub, const DevScratch* aux, const int* band, int cap, Best* partials,
              unsigned* ticket, lbm_angle* out) {
    const double qxc = aux->red.sx, qyc = aux->red.sy;
    const int nband = aux->band_n;
    Best b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) b[k] = Best{INFINITY, 0x7fffffffffffffffLL, 0, 0, 0};
    bool any = false;
    __shared__ long long s_id[4 * kRedThreads];
    __shared__ T s_va[4 * kRedThreads], s_vb[4 * kRedThreads];
    __shared__ int s_n;
    const bool listed = nband >= 0 && nband <= cap;
    const long long total = listed ? nband : (long long)nx * ny;
    const long long stride = (long long)gridDim.x * kRedThreads;
    for (long long first = (long long)blockIdx.x * kRedThreads; first < total; first += stride) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const long long t = first + threadIdx.x;
        unsigned m = 0;
        T va = 0, vb[4];
        int n = 0;
        if (t < total) {
            n = listed ? band[t] : (int)t;  // fewer than 2^31 nodes
            const int j = n / nx, i = n - j * nx;
            if (listed || flags[lidx(P, i, j)] == kFluid) {
                va = rho[lidx(P, i, j)];
                const unsigned ends = link_ends<T>(rho, flags, nx, ny, P, i, j, vb);
                m = listed ? crossing_links<T, true>(va, vb, ends, rho_m, thr, sub, i, j)
                           : crossing_links<T, false>(va, vb, ends, rho_m, thr, sub, i, j);
            }
        }
        if (m) {
            int at = atomicAdd(&s_n, __popc(m));
#pragma unroll
            for (int sl = 0; sl < 4; ++sl)
                if (m >> sl & 1) {
                    s_id[at] = (long long)n * 4 + sl;
                    s_va[at] = va;
                    s_vb[at] = vb[sl];
                    ++at;
                }
        }
        __syncthreads();
        for (int k = threadIdx.x; k < s_n; k += kRedThreads)
            any |= take_link<T>(s_id[k], nx, s_va[k], s_vb[k], rho_m, thr, sub, qxc, qyc, b);
        __syncthreads();
    }
    __shared__ Best s[kRedThreads / 32][4];
    __shared__ int s_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (__syncthreads_or(any)) {
        const bool warp_any = __any_sync(0xffffffffu, any);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (warp_any)
                for (int o = 16; o > 0; o >>= 1) shfl_best(b[k], o);
            if (lane == 0) s[warp][k] = b[k];
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            Best r = s[0][threadIdx.x];
            for (int w = 1; w < kRedThreads / 32; ++w)
                if (better(s[w][threadIdx.x].key, s[w][threadIdx.x].id, r.key, r.id))
                    r = s[w][threadIdx.x];
            partials[(size_t)blockIdx.x * 4 + threadIdx.x] = r;
        }
    } else if (threadIdx.x < 4) {
        partials[(size_t)blockIdx.x * 4 + threadIdx.x] =
            Best{INFINITY, 0x7fffffffffffffffLL, 0, 0, 0};
    }
    if (!last_block(ticket, gridDim.x, &s_last)) return;
    __shared__ Best win[4];
    if (warp < 4) {
        Best r = Best{INFINITY, 0x7fffffffffffffffLL, 0, 0, 0};
        for (int blk = lane; blk < (int)gridDim.x; blk += 32) {
            const Best* c = partials + (size_t)blk * 4 + warp;
            const double key = __ldcg(&c->key);
            if (!(key < INFINITY)) continue;
            const long long id = __ldcg(&c->id);
            if (better(key, id, r.key, r.id))
                r = Best{key, id, __ldcg(&c->px), __ldcg(&c->py), __ldcg(&c->d)};
        }
        for (int o = 16; o > 0; o >>= 1) shfl_best(r, o);
        if (lane == 0) win[warp] = r;
    }
    __syncthreads();
    __shared__ double s_alpha[2];
    const int side = warp & 1;
    lbm_angle o{};
    bool ok = false;
    if (warp < 4 && lane == 0) {
        double ct = 0, at = 0;
        ok = side_line(win[side * 2], win[side * 2 + 1], sub, side, &o, ct, at);
        if (ok && warp < 2) o.theta_deg = acos(ct) * (180.0 / M_PI);
        if (ok && warp >= 2) s_alpha[side] = acos(at) * (180.0 / M_PI);
    }
    __syncthreads();
    if (warp < 2 && lane == 0) {
        if (ok) {
            o.alpha_deg = s_alpha[side];
            o.beta_deg = !sub.circle ? o.theta_deg
                         : (sub.concave ? o.theta_deg - o.alpha_deg : o.theta_deg + o.alpha_deg);
        }
        out[side] = o;
    }
}

// dense per-(node, slot) candidate marks and points, for parity checks
template <typename T>
__global__ void k_cand_dense(const T* rho, const uint8_t* flags, int nx, int ny, int P,
                             double rho_m, T thr, Substrate sub, uint8_t* mark, double* pxyd) {
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < (long long)nx * ny;
         n += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(n / nx), i = (int)(n % nx);
        const bool fl = flags[lidx(P, i, j)] == kFluid;
        const T va = rho[lidx(P, i, j)];
        T vb[4];
        const unsigned ends = link_ends<T>(rho, flags, nx, ny, P, i, j, vb);
#pragma unroll
        for (int sl = 0; sl < 4; ++sl) {
            double px = 0, py = 0;
            const bool ok = fl && (ends >> sl & 1) &&
                            link_point<T>(va, vb[sl], rho_m, thr, i, j, sl, px, py);
            mark[n * 4 + sl] = ok ? 1 : 0;
            if (ok) {
                pxyd[(n * 4 + sl) * 3 + 0] = px;
                pxyd[(n * 4 + sl) * 3 + 1] = py;
                pxyd[(n * 4 + sl) * 3 + 2] = substrate_dist(sub, px, py);
            }
        }
    }
}

// Field out as doubles (0 at solid nodes), four nodes per thread when the rows of the destination allow
// it: 2^lt threads per row, as many as a row of nx nodes has groups of four (at most the block's 256),
// so that the index needs no division; a block takes 256 >> lt rows and 4 << lt columns. One row per
// block left most threads of a narrow lattice idle: 16 x 60000 46 us per read, 20 so.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    k_to_double(const T* src, const uint8_t* flags, int nx, int ny, int P, int lt, double* dst) {
    const int j = blockIdx.x * (kRedThreads >> lt) + (threadIdx.x >> lt);
    const int i0 = ((blockIdx.y << lt) + (threadIdx.x & ((1 << lt) - 1))) * 4;
    if (i0 >= nx || j >= ny) return;
    const int e = lidx(P, i0, j);
    const uint32_t f = __ldg(reinterpret_cast<const unsigned*>(flags + e));
    T r[4];
    load4(src + e, r);
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = ((f >> (8 * k)) & 0xFFu) == kFluid ? (double)r[k] : 0.0;
    double* o = dst + (size_t)j * nx + i0;
    if (i0 + 4 <= nx && ((uintptr_t)o & 15) == 0) {
        reinterpret_cast<double2*>(o)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2*>(o)[1] = make_double2(v[2], v[3]);
    } else {
        for (int k = 0; k < 4 && i0 + k < nx; ++k) o[k] = v[k];
    }
}

}  // namespace

size_t reduce_partial_bytes(int nblocks) { return 5 * sizeof(double) * (size_t)nblocks; }
size_t meas_partial_bytes(int nblocks) { return sizeof(Best) * 4 * (size_t)nblocks; }

// mapped host memory for the results, made at the first call that needs it
cudaError_t ensure_host_out(lbm_ctx* c) {
    if (c->host_out_dev) return cudaSuccess;
    if (!c->host_out) {
        void* h = nullptr;
        const cudaError_t e = cudaHostAlloc(&h, sizeof(HostOut), cudaHostAllocMapped);
        if (e != cudaSuccess) return e;
        c->host_out = (HostOut*)h;
    }
    void* d = nullptr;
    const cudaError_t e = cudaHostGetDevicePointer(&d, c->host_out, 0);
    if (e == cudaSuccess) c->host_out_dev = (HostOut*)d;
    return e;
}

namespace {

// the largest T that is not above x
float floor_to(double x, float) {
    const float f = (float)x;
    return (double)f > x ? nextafterf(f, -INFINITY) : f;
}
double floor_to(double x, double) { return x; }

template <typename T>
cudaError_t reduce_t(lbm_ctx* c, ReduceOut* host) {
    const double rho_m = 0.5 * (c->rho_g + c->rho_l);
    int lt = 0;
    while ((1 << lt) < kRedThreads) ++lt;
    while (lt > 0 && c->ny > (long long)c->red_blocks * (kRedThreads >> lt) && 8 << (lt - 1) >= c->nx) --lt;
    Partials p;
    p.mass = (double*)c->red_partials;
    p.cnt = (unsigned long long*)(p.mass + c->red_blocks);
    k_reduce<T><<<c->red_blocks, kRedThreads, 0, c->stream>>>(
        (const T*)c->rho[c->cur], c->flags, c->nx, c->ny, c->P, lt, floor_to(rho_m, T()), p,
        &c->aux->ticket[0], &c->aux->red, host);
    return cudaGetLastError();
}

template <typename T>
cudaError_t measure_t(lbm_ctx* c) {
    const double rho_m = 0.5 * (c->rho_g + c->rho_l);
    k_measure<T><<<c->meas_blocks, kRedThreads, 0, c->stream>>>(
        (const T*)c->rho[c->cur], c->flags, c->nx, c->ny, c->P, rho_m, floor_to(rho_m, T()), c->sub,
        c->aux, c->band,
        c->band_cap, (Best*)c->meas_partials, &c->aux->ticket[1], c->host_out_dev->angle);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_reduce(lbm_ctx* c, bool to_host) {
    ReduceOut* host = to_host ? &c->host_out_dev->red : nullptr;
    return c->esz == 4 ? reduce_t<float>(c, host) : reduce_t<double>(c, host);
}

cudaError_t launch_measure(lbm_ctx* c) {
    const cudaError_t e = launch_reduce(c, false);
    if (e != cudaSuccess) return e;
    return c->esz == 4 ? measure_t<float>(c) : measure_t<double>(c);
}

cudaError_t launch_candidates(lbm_ctx* c, uint8_t* d_mark, double* d_pxyd) {
    const double rho_m = 0.5 * (c->rho_g + c->rho_l);
    const int blocks = 2 * c->sms;  // (not a block per row: wide, flat lattices have few)
    if (c->esz == 4)
        k_cand_dense<float><<<blocks, kRedThreads, 0, c->stream>>>(
            (const float*)c->rho[c->cur], c->flags, c->nx, c->ny, c->P, rho_m,
            floor_to(rho_m, 0.f), c->sub, d_mark,
            d_pxyd);
    else
        k_cand_dense<double><<<blocks, kRedThreads, 0, c->stream>>>(
            (const double*)c->rho[c->cur], c->flags, c->nx, c->ny, c->P, rho_m, rho_m, c->sub, d_mark,
            d_pxyd);
    return cudaGetLastError();
}

cudaError_t launch_to_double(lbm_ctx* c, const void* src, double* dst, int) {
    int lt = 0;
    while ((1 << lt) < kRedThreads && (4 << lt) < c->nx) ++lt;
    const int rows = kRedThreads >> lt;
    // rows along x (2^20 of them at most), column blocks along y
    const dim3 grid((c->ny + rows - 1) / rows, (c->nx + (4 << lt) - 1) / (4 << lt));
    if (c->esz == 4)
        k_to_double<float><<<grid, kRedThreads, 0, c->stream>>>((const float*)src, c->flags, c->nx, c->ny,
                                                                c->P, lt, dst);
    else
        k_to_double<double><<<grid, kRedThreads, 0, c->stream>>>((const double*)src, c->flags, c->nx,
                                                                 c->ny, c->P, lt, dst);
    return cudaGetLastError();
}

}  // namespace lbm

// Objective evaluation of a reconstruction against sensor views (Sec. III-E).
//
// Geometry (eq. (3)-(5)), for one view with the rendered depth D_r and the
// sensor depth D_g (0 = background; silhouettes S_r = D_r > 0, S_g = D_g > 0):
//   k_ev_cols    the vertical distance of every pixel to the nearest pixel of
//                S_g and of S_r in its column, and the counts |S_r|, |S_g|,
//                |xor|, |or|: a warp reads 32 rows of 32 columns into one bit
//                mask per column and set, the distances come from the masks;
//   k_ev_rows    one CTA per row: for each pixel of S_r the exact squared
//                distance to S_g, min over columns x' of (x - x')^2 + col(x')^2
//                (searched outwards, stopped once (x - x')^2 exceeds the best),
//                and the same from S_g to S_r; the maxima (eq. (4)) by
//                atomicMax -- integers throughout, so exact;
//   k_ev_points  one CTA per 16 x 16 pixels: back-projects the foreground
//                pixels, X = z (dx, dy, 1), into two lists (a tile's points
//                are contiguous; the order of the tiles does not matter) and
//                records the box of the tile's rendered points;
//   k_ev_cp      per sensor point the squared distance to the closest rendered
//                point, float32: only 8 x 8 pixel blocks whose box can hold a
//                closer point than the best so far are searched;
//   k_sum / k_sum_final  the float64 sum of those distances in pixel order,
//                fixed blocks and a fixed tree (deterministic).
//
// Appearance (eq. (6)(7)), per scale j = 1..3:
//   k_ap_luma / k_ap_down   luma planes and silhouette, then 2 x 2 block
//                mean (silhouette: block AND) for the next scale;
//   k_ap_ssim    32 x 16 pixels per CTA with an 11 x 11-window halo in shared
//                memory: per silhouette pixel the window means, then the
//                second moments about those means (centred, so flat regions
//                give exactly zero variance up to rounding of the mean),
//                l, c, s and w(u); block partial sums in float64;
//   k_ap_final   the partials of every scale and term in a fixed order.
// The host side combines the per-scale means into WMS3IM.
#include <cuda_runtime.h>
#include <math.h>

#include <limits>
#include <mutex>
#include <set>

#include "ftr_internal.h"

namespace ftr {

namespace {

constexpr int kNone = 1 << 28;      // column distance when the column holds no pixel of the set
constexpr long long kFar = 0x7fffffffffffffffLL;   // no pixel of the set in the whole image
constexpr int kTile = 16;           // closest points: pixels per tile side
constexpr int kR = 5;               // SSIM window radius (11 x 11)
constexpr int kSsimW = 32, kSsimH = 16;                                  // SSIM: output pixels per CTA
constexpr int kHaloW = kSsimW + 2 * kR, kHaloH = kSsimH + 2 * kR;
constexpr int kSumBlocks = 256;
constexpr int kCpThreads = 64;      // closest points: small CTAs, so that one body's points reach every SM
// counters of one geometry evaluation: |S_r|, |S_g|, |xor|, |or|, the two
// squared Hausdorff maxima, the list sizes I and J, the tiles with rendered
// points, the float64 sum of the closest-point distances, and the entries of
// the sensor list (whole warps)
constexpr int kCounters = 11;
// Sec. III-E3: exponents of the three scales (luminance, contrast, structure)
constexpr double kAlpha[3] = {0.0, 0.0, 0.1333};
constexpr double kBeta[3] = {0.0448, 0.3001, 0.1333};
constexpr double kGamma[3] = {0.0448, 0.3001, 0.1333};

struct Taps {
    float g[2 * kR + 1];
};

// Distance of row y = base + i to the nearest set row of its column: m = the
// column's mask of rows base .. base + 31, prev / next = the nearest set rows
// of the segments before and after (-1: none).
__device__ __forceinline__ int col_distance(unsigned m, int i, int base, int prev, int next) {
    const unsigned upto = m & (0xffffffffu >> (31 - i)), from = m >> i;
    const int last = upto ? base + 31 - __clz(upto) : prev;
    const int nxt = from ? base + i + __ffs(from) - 1 : next;
    int d = kNone;
    if (last >= 0) d = base + i - last;
    if (nxt >= 0) d = min(d, nxt - (base + i));
    return d;
}

// One CTA per 32 columns, a warp per 32-row segment (grid-stride over the
// segments): the segment's rows are loaded at once and kept as one bit per row
// and set, so the column is read once and its distances need no second sweep.
// (A thread per column walking all rows twice ran 4 CTAs for a 512-pixel row
// and took 380 us at 512 x 424, all of it dependent loads; now 12.)  Shared memory:
// masks [set][segment][column], 256 bytes per segment.
__global__ void __launch_bounds__(512) k_ev_cols(const float* __restrict__ rd, const float* __restrict__ gd, int w,
                                                 int h, int nseg, int* __restrict__ colG, int* __restrict__ colR,
                                                 unsigned long long* __restrict__ cnt) {
    extern __shared__ unsigned s_m[];
    unsigned* s_g = s_m;
    unsigned* s_r = s_m + nseg * 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int x = blockIdx.x * 32 + lane;
    unsigned nr = 0, ng = 0, nx = 0, no = 0;
    for (int s = wid; s < nseg; s += nw) {
        unsigned mg = 0, mr = 0;
        if (x < w) {
            const int64_t at = (int64_t)s * 32 * w + x;
            const int rows = h - s * 32;            // all loads of 16 rows in flight at once
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += 16) {
                float vg[16], vr[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    vg[i] = i0 + i < rows ? gd[at + (int64_t)(i0 + i) * w] : 0.f;
                    vr[i] = i0 + i < rows ? rd[at + (int64_t)(i0 + i) * w] : 0.f;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    mg |= (unsigned)(vg[i] > 0.f) << (i0 + i);
                    mr |= (unsigned)(vr[i] > 0.f) << (i0 + i);
                }
            }
        }
        s_g[s * 32 + lane] = mg;
        s_r[s * 32 + lane] = mr;
        nr += __popc(mr);
        ng += __popc(mg);
        nx += __popc(mr ^ mg);
        no += __popc(mr | mg);
    }
    __syncthreads();
    if (x < w) {
        for (int s = wid; s < nseg; s += nw) {
            int pg = -1, pr = -1, qg = -1, qr = -1;
            for (int t = s - 1; t >= 0 && pg < 0; --t)
                if (s_g[t * 32 + lane]) pg = t * 32 + 31 - __clz(s_g[t * 32 + lane]);
            for (int t = s - 1; t >= 0 && pr < 0; --t)
                if (s_r[t * 32 + lane]) pr = t * 32 + 31 - __clz(s_r[t * 32 + lane]);
            for (int t = s + 1; t < nseg && qg < 0; ++t)
                if (s_g[t * 32 + lane]) qg = t * 32 + __ffs(s_g[t * 32 + lane]) - 1;
            for (int t = s + 1; t < nseg && qr < 0; ++t)
                if (s_r[t * 32 + lane]) qr = t * 32 + __ffs(s_r[t * 32 + lane]) - 1;
            const unsigned mg = s_g[s * 32 + lane], mr = s_r[s * 32 + lane];
            const int rows = min(32, h - s * 32);
#pragma unroll 4
            for (int i = 0; i < rows; ++i) {
                const int64_t at = (int64_t)(s * 32 + i) * w + x;
                colG[at] = col_distance(mg, i, s * 32, pg, qg);
                colR[at] = col_distance(mr, i, s * 32, pr, qr);
            }
        }
    }
    nr = __reduce_add_sync(0xffffffffu, nr);
    ng = __reduce_add_sync(0xffffffffu, ng);
    nx = __reduce_add_sync(0xffffffffu, nx);
    no = __reduce_add_sync(0xffffffffu, no);
    if (lane == 0 && no) {
        atomicAdd(cnt + 0, (unsigned long long)nr);
        atomicAdd(cnt + 1, (unsigned long long)ng);
        atomicAdd(cnt + 2, (unsigned long long)nx);
        atomicAdd(cnt + 3, (unsigned long long)no);
    }
}

// Smallest (x - x')^2 + col(x')^2 over the row; kNone columns hold no pixel.
__device__ __forceinline__ long long row_min(const int* __restrict__ col, int w, int x) {
    long long best = kFar;
    for (int d = 0; d < w; ++d) {
        const long long dd = (long long)d * d;
        if (dd >= best) break;
        if (x - d >= 0) {
            const int c = col[x - d];
            if (c != kNone) best = min(best, dd + (long long)c * c);
        }
        if (d > 0 && x + d < w) {
            const int c = col[x + d];
            if (c != kNone) best = min(best, dd + (long long)c * c);
        }
    }
    return best;
}

__global__ void __launch_bounds__(256) k_ev_rows(const float* __restrict__ rd, const float* __restrict__ gd, int w,
                                                 const int* __restrict__ colG, const int* __restrict__ colR,
                                                 unsigned long long* __restrict__ cnt) {
    const int y = blockIdx.x;
    const int64_t row = (int64_t)y * w;
    unsigned long long mrg = 0, mgr = 0;
    for (int x = threadIdx.x; x < w; x += blockDim.x) {
        if (rd[row + x] > 0.f) {
            const long long b = row_min(colG + row, w, x);
            if (b != kFar) mrg = max(mrg, (unsigned long long)b);
        }
        if (gd[row + x] > 0.f) {
            const long long b = row_min(colR + row, w, x);
            if (b != kFar) mgr = max(mgr, (unsigned long long)b);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mrg = max(mrg, __shfl_xor_sync(0xffffffffu, mrg, o));
        mgr = max(mgr, __shfl_xor_sync(0xffffffffu, mgr, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (mrg) atomicMax(cnt + 4, mrg);
        if (mgr) atomicMax(cnt + 5, mgr);
    }
}

struct Intr {
    double K[9];
};

// Rendered points of one 8 x 8 pixel block: their bounding box and their place
// in the list.  A 16 x 16 pixel tile holds four of them and the box of all.
struct PointBox {
    float lo[3];
    int start;
    float hi[3];
    int count;
};
struct PointTile {
    PointBox all, part[4];
};

// A warp takes 8 x 4 pixels and a pair of warps one 8 x 8 block, so that a
// block's points are near one another.  The sensor points of a warp that has
// any keep a whole warp's entries (the rest repeat one of them, tag -1): a warp
// of k_ev_cp then never holds the points of two distant patches.  tile_of: per
// image tile its record, -1 without rendered points.
__global__ void __launch_bounds__(256) k_ev_points(const float* __restrict__ rd, const float* __restrict__ gd,
                                                   int w, int h, Intr in, float4* __restrict__ ptsG,
                                                   float4* __restrict__ ptsR, PointTile* __restrict__ tiles,
                                                   int* __restrict__ tile_of, float* __restrict__ d2,
                                                   unsigned long long* __restrict__ cnt) {
    __shared__ int s_ng[8], s_nr[8], s_base[3];
    __shared__ float s_box[8][6];
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int x = blockIdx.x * kTile + ((wid >> 1) & 1) * 8 + (lane & 7);
    const int y = blockIdx.y * kTile + (wid >> 2) * 8 + (wid & 1) * 4 + (lane >> 3);
    const bool live = x < w && y < h;
    const int64_t p = (int64_t)y * w + x;
    const float zg = live ? gd[p] : 0.f, zr = live ? rd[p] : 0.f;
    const bool g = zg > 0.f, r = zr > 0.f;
    int* own = tile_of + (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
    if (live) d2[p] = g ? __uint_as_float(0x7f800000u) : 0.f;
    if (!__syncthreads_or(g || r)) {
        if (threadIdx.x == 0) *own = -1;
        return;
    }
    double dx = 0.0, dy = 0.0;
    if (g || r) {
        const double py = (double)y, px = (double)x;
        dy = __ddiv_rn(__dsub_rn(py, in.K[5]), in.K[4]);
        dx = __ddiv_rn(__dsub_rn(__dsub_rn(px, in.K[2]), __dmul_rn(in.K[1], dy)), in.K[0]);
    }
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
    const float inf = __uint_as_float(0x7f800000u);
    float b[6] = {inf, inf, inf, -inf, -inf, -inf};
    if (r) {
        const double z = zr;
        P = make_float4((float)(z * dx), (float)(z * dy), zr, __int_as_float((int)p));
        b[0] = fminf(inf, P.x);               // a NaN coordinate leaves the box as it is
        b[1] = fminf(inf, P.y);
        b[2] = fminf(inf, P.z);
        b[3] = fmaxf(-inf, P.x);
        b[4] = fmaxf(-inf, P.y);
        b[5] = fmaxf(-inf, P.z);
    }
    const unsigned lt = (1u << lane) - 1u;
    const unsigned bg = __ballot_sync(0xffffffffu, g), br = __ballot_sync(0xffffffffu, r);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            b[c] = fminf(b[c], __shfl_xor_sync(0xffffffffu, b[c], o));
            b[3 + c] = fmaxf(b[3 + c], __shfl_xor_sync(0xffffffffu, b[3 + c], o));
        }
    }
    if (lane == 0) {
        s_ng[wid] = __popc(bg);
        s_nr[wid] = __popc(br);
#pragma unroll
        for (int c = 0; c < 6; ++c) s_box[wid][c] = b[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int ng = 0, nr = 0, slots = 0;
        for (int k = 0; k < 8; ++k) {
            ng += s_ng[k];
            nr += s_nr[k];
            slots += s_ng[k] ? 32 : 0;
        }
        if (ng) atomicAdd(cnt + 6, (unsigned long long)ng);
        s_base[0] = ng ? (int)atomicAdd(cnt + 10, (unsigned long long)slots) : 0;
        s_base[1] = nr ? (int)atomicAdd(cnt + 7, (unsigned long long)nr) : 0;
        s_base[2] = nr ? (int)atomicAdd(cnt + 8, 1ull) : -1;
        *own = s_base[2];
    }
    __syncthreads();
    if (s_base[2] >= 0 && threadIdx.x < 5) {      // the tile's record: thread 4 the whole, 0..3 the blocks
        const int k0 = threadIdx.x == 4 ? 0 : 2 * threadIdx.x, k1 = threadIdx.x == 4 ? 8 : k0 + 2;
        PointBox t;
        t.start = s_base[1];
        for (int k = 0; k < k0; ++k) t.start += s_nr[k];
        t.count = 0;
        for (int c = 0; c < 3; ++c) {
            t.lo[c] = inf;
            t.hi[c] = -inf;
        }
        for (int k = k0; k < k1; ++k) {
            t.count += s_nr[k];
            for (int c = 0; c < 3; ++c) {
                t.lo[c] = fminf(t.lo[c], s_box[k][c]);
                t.hi[c] = fmaxf(t.hi[c], s_box[k][3 + c]);
            }
        }
        if (threadIdx.x == 4)
            tiles[s_base[2]].all = t;
        else
            tiles[s_base[2]].part[threadIdx.x] = t;
    }
    int og = s_base[0], orr = s_base[1];
    for (unsigned k = 0; k < wid; ++k) {
        og += s_ng[k] ? 32 : 0;
        orr += s_nr[k];
    }
    if (bg) {
        float4 Q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g) {
            const double z = zg;
            Q = make_float4((float)(z * dx), (float)(z * dy), zg, 0.f);
        }
        const int first = __ffs(bg) - 1;
        const float fx = __shfl_sync(0xffffffffu, Q.x, first), fy = __shfl_sync(0xffffffffu, Q.y, first),
                    fz = __shfl_sync(0xffffffffu, Q.z, first);
        ptsG[og + lane] = g ? make_float4(Q.x, Q.y, Q.z, __int_as_float((int)p))
                            : make_float4(fx, fy, fz, __int_as_float(-1));
    }
    if (r) ptsR[orr + __popc(br & lt)] = P;
}

// Squared distance from a box (or a point, lo = hi) to a box, not above that of
// any two points in them (differences and sums of float32 are monotonic; the
// factor covers the order the sum is rounded in).
__device__ __forceinline__ float box_gap2(const float lo[3], const float hi[3], const PointBox& b) {
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float d = fmaxf(fmaxf(b.lo[c] - hi[c], lo[c] - b.hi[c]), 0.f);
        s += d * d;
    }
    return s * 0.9999f;
}

// Per sensor point the squared distance to the closest rendered point: the
// minimum over all of them, found by searching only the blocks whose box can
// hold a closer point, so the result is that of the full search.  A warp holds
// the points of one 8 x 4 pixel patch and searches together: its own tile
// first, which leaves most lanes with the distance to the surface (where that
// is empty, the tile whose farthest corner is nearest); then its lanes test 32
// tile boxes at a time against the box of the warp's points, and the blocks of
// those that remain per lane.  28,000 x 28,000 points of a 512 x 424 view: 107
// us for all pairs, 94 with 16 x 16 tiles tested lane by lane in list order, 55
// now; the last warps, whose patch lies off the rendered silhouette, decide it.
__global__ void __launch_bounds__(kCpThreads) k_ev_cp(const float4* __restrict__ G, const float4* __restrict__ R,
                                                      const PointTile* __restrict__ tiles,
                                                      const int* __restrict__ tile_of, int w,
                                                      const unsigned long long* __restrict__ cnt,
                                                      float* __restrict__ d2) {
    const int nt = (int)cnt[8];
    const int64_t gi = (int64_t)blockIdx.x * kCpThreads + threadIdx.x;
    if (gi >= (int64_t)cnt[10]) return;                    // whole warps
    const unsigned lane = threadIdx.x & 31;
    const float inf = __uint_as_float(0x7f800000u);
    const float4 q = G[gi];
    const int tag = __float_as_int(q.w);                   // pixel, -1: a repeated point
    float best = inf, bound = inf;
    auto search = [&](const PointBox& b) {
        const float4* pr = R + b.start;
#pragma unroll 8
        for (int k = 0; k < b.count; ++k) {
            const float4 c = __ldg(pr + k);
            const float ex = q.x - c.x, ey = q.y - c.y, ez = q.z - c.z;
            best = fminf(best, ex * ex + ey * ey + ez * ez);
        }
    };
    const float ql[3] = {q.x, q.y, q.z};
    auto visit = [&](const PointTile& t) {                 // warp-uniform
        for (int s = 0; s < 4; ++s) {
            const bool want = !(box_gap2(ql, ql, t.part[s]) > fminf(best, bound));
            if (t.part[s].count > 0 && __any_sync(0xffffffffu, want)) search(t.part[s]);
        }
    };
    // the tile of the warp's points
    const int p0 = __reduce_max_sync(0xffffffffu, tag);
    const int own = tile_of[(int64_t)(p0 / w / kTile) * ((w + kTile - 1) / kTile) + (p0 % w) / kTile];
    if (own >= 0) visit(tiles[own]);
    float lo[3], hi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) lo[c] = hi[c] = ql[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
    }
    float reach;                                           // no lane looks farther
    auto update_reach = [&]() {
        reach = fminf(best, bound);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) reach = fmaxf(reach, __shfl_xor_sync(0xffffffffu, reach, o));
    };
    update_reach();
    if (reach == inf) {
        float far = inf;                                   // farthest corners of the two boxes
        int at = -1;
        for (int j = lane; j < nt; j += 32) {
            const PointBox b = tiles[j].all;
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float d = fmaxf(fabsf(b.hi[c] - lo[c]), fabsf(hi[c] - b.lo[c]));
                s += d * d;
            }
            if (s * 1.0001f < far) {
                far = s * 1.0001f;
                at = j;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float of = __shfl_xor_sync(0xffffffffu, far, o);
            const int oa = __shfl_xor_sync(0xffffffffu, at, o);
            if (of < far || (of == far && oa > at)) {      // the same choice in every lane
                far = of;
                at = oa;
            }
        }
        bound = far;
        if (at >= 0) visit(tiles[at]);
        update_reach();
    }
    for (int jb = 0; jb < nt; jb += 32) {
        const int j = jb + (int)lane;
        bool want = false;
        if (j < nt && j != own) {
            const PointBox b = tiles[j].all;
            want = !(box_gap2(lo, hi, b) > reach);
        }
        unsigned m = __ballot_sync(0xffffffffu, want);
        while (m) {
            const int k = jb + __ffs(m) - 1;
            m &= m - 1;
            visit(tiles[k]);
        }
        update_reach();
    }
    if (tag >= 0) d2[tag] = best;
}

// float64 sums of n values in a fixed order: block b takes the indices
// b*256 + t + k*gridDim*256, then a fixed tree.
template <class T>
__global__ void __launch_bounds__(256) k_sum(const T* __restrict__ v, int64_t n, double* __restrict__ part) {
    __shared__ double s[256];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) acc += (double)v[i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

// The block sums in a fixed order.
__global__ void __launch_bounds__(256) k_sum_final(const double* __restrict__ part, int64_t nblocks,
                                                   double* __restrict__ out) {
    __shared__ double s[256];
    double acc = 0.0;
    for (int64_t b = threadIdx.x; b < nblocks; b += 256) acc += part[b];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = s[0];
}

__global__ void __launch_bounds__(256) k_ap_luma(const uint8_t* __restrict__ rr, const uint8_t* __restrict__ rg,
                                                 const float* __restrict__ rd, int64_t npx, float* __restrict__ X,
                                                 float* __restrict__ Y, uint8_t* __restrict__ S) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npx) return;
    X[p] = 0.299f * rr[3 * p] + 0.587f * rr[3 * p + 1] + 0.114f * rr[3 * p + 2];
    Y[p] = 0.299f * rg[3 * p] + 0.587f * rg[3 * p + 1] + 0.114f * rg[3 * p + 2];
    S[p] = rd[p] > 0.f;
}

__global__ void __launch_bounds__(256) k_ap_down(const float* __restrict__ X, const float* __restrict__ Y,
                                                 const uint8_t* __restrict__ S, int w, int w2, int h2,
                                                 float* __restrict__ X2, float* __restrict__ Y2,
                                                 uint8_t* __restrict__ S2) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)w2 * h2) return;
    const int64_t y = p / w2, x = p % w2;
    const int64_t a = 2 * y * w + 2 * x, b = a + w;
    X2[p] = 0.25f * (((X[a] + X[a + 1]) + X[b]) + X[b + 1]);
    Y2[p] = 0.25f * (((Y[a] + Y[a + 1]) + Y[b]) + Y[b + 1]);
    S2[p] = S[a] & S[a + 1] & S[b] & S[b + 1];
}

// The SSIM terms of one pixel from its window moments, times the window's
// silhouette count.
struct SsimSums {
    double l, c, s, w;
};

__device__ __forceinline__ void ssim_terms(float mx, float my, float vx, float vy, float cxy, int count, SsimSums& a) {
    const float C1 = (0.01f * 255.f) * (0.01f * 255.f);
    const float C2 = (0.03f * 255.f) * (0.03f * 255.f);
    const float C3 = 0.5f * C2;
    const float sgx = sqrtf(vx), sgy = sqrtf(vy);
    const float l = (2.f * mx * my + C1) / (mx * mx + my * my + C1);
    const float c = (2.f * sgx * sgy + C2) / (vx + vy + C2);
    const float s = (cxy + C3) / (sgx * sgy + C3);
    const double cw = (double)count;
    a.l += cw * l;
    a.c += cw * c;
    a.s += cw * s;
    a.w += cw;
}

// A thread takes two vertically adjacent pixels of a 32 x 16 tile.  The window
// means are separable and keep the order of the direct sums: the row sums of
// the 26 x 32 halo rows are formed once in shared memory and each pixel adds
// its 11.  The second moments stay centred on each pixel's own mean (an
// expansion about a common point would cancel in flat regions), so their 121
// samples are read once for the two pixels.  A tile without silhouette pixels
// ends after its loads; a tile that touches the image border takes the windows
// cut at it.  (16 x 16 pixels with direct, bounds-tested 121-tap sums for the
// means and the moments ran 182 + 137 + 57 us for the three scales of a 1920 x
// 1080 view whose silhouette covers an eighth of it.)  One launch for the tiles of
// all scales: each scale's last tiles are a dependent chain of some 10 us that the
// others now cover (26 + 23 + 11 us one after another, now 34).
struct ApScales {
    int64_t at[4];            // first tile (= partial of 4 terms) of each scale, and their number
    int64_t plane[3];         // first pixel of each scale in X, Y and S
    int w[3], h[3], gx[3];    // pixels, tiles per row
};

__global__ void __launch_bounds__(256) k_ap_ssim(const float* __restrict__ Xs, const float* __restrict__ Ys,
                                                 const uint8_t* __restrict__ Ss, const __grid_constant__ ApScales sc,
                                                 const __grid_constant__ Taps tp, double* __restrict__ part) {
    __shared__ float sx[kHaloH][kHaloW];
    __shared__ float sy[kHaloH][kHaloW];
    __shared__ uint8_t ss[kHaloH][kHaloW + 2];
    __shared__ float rowx[kHaloH][kSsimW];
    __shared__ float rowy[kHaloH][kSsimW];
    __shared__ int rown[kHaloH][kSsimW];
    __shared__ double red[4][8];
    const int j3 = (int64_t)blockIdx.x < sc.at[1] ? 0 : ((int64_t)blockIdx.x < sc.at[2] ? 1 : 2);
    const float* X = Xs + sc.plane[j3];
    const float* Y = Ys + sc.plane[j3];
    const uint8_t* S = Ss + sc.plane[j3];
    const int w = sc.w[j3], h = sc.h[j3];
    const int tile = (int)(blockIdx.x - sc.at[j3]), tile_y = tile / sc.gx[j3], tile_x = tile - tile_y * sc.gx[j3];
    const int bx = tile_x * kSsimW - kR, by = tile_y * kSsimH - kR;
    const int tx = threadIdx.x % kSsimW, ty = 2 * (threadIdx.x / kSsimW);
    const int x = tile_x * kSsimW + tx, y = tile_y * kSsimH + ty;
    double* out = part + 4 * (int64_t)blockIdx.x;
    const bool in0 = x < w && y < h && S[(int64_t)y * w + x];
    const bool in1 = x < w && y + 1 < h && S[(int64_t)(y + 1) * w + x];
    if (!__syncthreads_or(in0 || in1)) {
        if (threadIdx.x < 4) out[threadIdx.x] = 0.0;
        return;
    }
    for (int i = threadIdx.x; i < kHaloH * kHaloW; i += 256) {
        const int hy = i / kHaloW, hx = i % kHaloW;
        const int gx = bx + hx, gy = by + hy;
        const bool in = gx >= 0 && gx < w && gy >= 0 && gy < h;
        const int64_t gi = (int64_t)gy * w + gx;
        sx[hy][hx] = in ? X[gi] : 0.f;
        sy[hy][hx] = in ? Y[gi] : 0.f;
        ss[hy][hx] = in ? S[gi] : 0;
    }
    __syncthreads();
    const bool inner = bx >= 0 && by >= 0 && bx + kHaloW <= w && by + kHaloH <= h;   // block-uniform
    for (int i = threadIdx.x; i < kHaloH * kSsimW; i += 256) {
        const int hy = i / kSsimW, hx = i % kSsimW;
        float rx = 0.f, ry = 0.f;
        int n = 0;
        if (inner) {
#pragma unroll
            for (int k = 0; k <= 2 * kR; ++k) {
                rx += tp.g[k] * sx[hy][hx + k];
                ry += tp.g[k] * sy[hy][hx + k];
                n += ss[hy][hx + k];
            }
        } else {
            const int gx = tile_x * kSsimW + hx;
            for (int k = max(0, kR - gx); k <= min(2 * kR, kR + w - 1 - gx); ++k) {
                rx += tp.g[k] * sx[hy][hx + k];
                ry += tp.g[k] * sy[hy][hx + k];
                n += ss[hy][hx + k];
            }
        }
        rowx[hy][hx] = rx;
        rowy[hy][hx] = ry;
        rown[hy][hx] = n;
    }
    __syncthreads();
    SsimSums a = {0.0, 0.0, 0.0, 0.0};
    if (inner) {
        if (in0 || in1) {
            float gsum = 0.f;
#pragma unroll
            for (int k = 0; k <= 2 * kR; ++k) gsum += tp.g[k];
            const float inv = 1.f / (gsum * gsum);
            float mx[2] = {0.f, 0.f}, my[2] = {0.f, 0.f};
            int n[2] = {0, 0};
#pragma unroll
            for (int j = 0; j <= 2 * kR + 1; ++j) {
                const float rx = rowx[ty + j][tx], ry = rowy[ty + j][tx];
                const int rn = rown[ty + j][tx];
                if (j <= 2 * kR) {
                    mx[0] += tp.g[j] * rx;
                    my[0] += tp.g[j] * ry;
                    n[0] += rn;
                }
                if (j >= 1) {
                    mx[1] += tp.g[j - 1] * rx;
                    my[1] += tp.g[j - 1] * ry;
                    n[1] += rn;
                }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                mx[q] *= inv;
                my[q] *= inv;
            }
            float vx[2] = {0.f, 0.f}, vy[2] = {0.f, 0.f}, cxy[2] = {0.f, 0.f};
#pragma unroll 1
            for (int j = 0; j <= 2 * kR + 1; ++j) {
                float ax[2] = {0.f, 0.f}, ay[2] = {0.f, 0.f}, axy[2] = {0.f, 0.f};
#pragma unroll
                for (int k = 0; k <= 2 * kR; ++k) {
                    const float g = tp.g[k], px = sx[ty + j][tx + k], py = sy[ty + j][tx + k];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float ex = px - mx[q], ey = py - my[q];
                        ax[q] += g * ex * ex;
                        ay[q] += g * ey * ey;
                        axy[q] += g * ex * ey;
                    }
                }
                if (j <= 2 * kR) {
                    vx[0] += tp.g[j] * ax[0];
                    vy[0] += tp.g[j] * ay[0];
                    cxy[0] += tp.g[j] * axy[0];
                }
                if (j >= 1) {
                    vx[1] += tp.g[j - 1] * ax[1];
                    vy[1] += tp.g[j - 1] * ay[1];
                    cxy[1] += tp.g[j - 1] * axy[1];
                }
            }
            if (in0) ssim_terms(mx[0], my[0], vx[0] * inv, vy[0] * inv, cxy[0] * inv, n[0], a);
            if (in1) ssim_terms(mx[1], my[1], vx[1] * inv, vy[1] * inv, cxy[1] * inv, n[1], a);
        }
    } else {
        for (int q = 0; q < 2; ++q) {
            if (!(q ? in1 : in0)) continue;
            // taps inside the image: columns i0..i1, rows j0..j1 of the window
            const int yq = y + q, tq = ty + q;
            const int i0 = max(0, kR - x), i1 = min(2 * kR, kR + w - 1 - x);
            const int j0 = max(0, kR - yq), j1 = min(2 * kR, kR + h - 1 - yq);
            float gsx = 0.f, gsy = 0.f;
            for (int i = i0; i <= i1; ++i) gsx += tp.g[i];
            for (int j = j0; j <= j1; ++j) gsy += tp.g[j];
            const float inv = 1.f / (gsx * gsy);
            float mx = 0.f, my = 0.f;
            int n = 0;
            for (int j = j0; j <= j1; ++j) {
                mx += tp.g[j] * rowx[tq + j][tx];
                my += tp.g[j] * rowy[tq + j][tx];
                n += rown[tq + j][tx];
            }
            mx *= inv;
            my *= inv;
            float vx = 0.f, vy = 0.f, cxy = 0.f;
            for (int j = j0; j <= j1; ++j) {
                float ax = 0.f, ay = 0.f, axy = 0.f;
                for (int i = i0; i <= i1; ++i) {
                    const float g = tp.g[i];
                    const float ex = sx[tq + j][tx + i] - mx, ey = sy[tq + j][tx + i] - my;
                    ax += g * ex * ex;
                    ay += g * ey * ey;
                    axy += g * ex * ey;
                }
                vx += tp.g[j] * ax;
                vy += tp.g[j] * ay;
                cxy += tp.g[j] * axy;
            }
            ssim_terms(mx, my, vx * inv, vy * inv, cxy * inv, n, a);
        }
    }
    double v[4] = {a.l, a.c, a.s, a.w};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[m] += __shfl_xor_sync(0xffffffffu, v[m], o);
        if ((threadIdx.x & 31) == 0) red[m][threadIdx.x >> 5] = v[m];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += red[threadIdx.x][k];
        out[threadIdx.x] = t;
    }
}

// The twelve sums of the three scales, one CTA each: CTA 4 j + m adds term m of
// scale j over that scale's tiles in a fixed order.
__global__ void __launch_bounds__(256) k_ap_final(const double* __restrict__ part, ApScales sc,
                                                  double* __restrict__ out) {
    __shared__ double s[8];
    const int j = blockIdx.x >> 2, m = blockIdx.x & 3;
    const double* p = part + 4 * sc.at[j] + m;
    double acc = 0.0;
#pragma unroll 8
    for (int64_t b = threadIdx.x; b < sc.at[j + 1] - sc.at[j]; b += 256) acc += p[4 * b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += s[k];
        out[blockIdx.x] = t;
    }
}

bool dev_ptr(const void* p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Shared memory of k_ev_cols for an image of h rows.
size_t col_smem(int h) { return (size_t)((h + 31) / 32) * 64 * sizeof(unsigned); }

// The limit belongs to the function on the device, for every context and host
// thread: raised once, to the largest image's 128 KB, and never lowered between
// another thread's check and its launch.
cudaError_t allow_col_smem(int device) {
    static std::mutex mu;
    static std::set<int> done;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count(device)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_ev_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)col_smem(16384));
    if (e == cudaSuccess) done.insert(device);
    return e;
}

template <class T>
cudaError_t grow(T** p, int64_t* cap, int64_t need) {
    if (*cap >= need) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    cudaError_t e = cudaMalloc((void**)p, (size_t)need * sizeof(T));
    if (e == cudaSuccess) *cap = need;
    return e;
}

cudaError_t grow_pixels(ftr_ctx* c, EvalScratch* ev, int64_t npx) {
    if (ev->pix_cap >= npx) return cudaSuccess;
    cudaStreamSynchronize(c->stream);
    if (ev->col) cudaFree(ev->col);
    if (ev->pts) cudaFree(ev->pts);
    if (ev->d2) cudaFree(ev->d2);
    ev->col = nullptr;
    ev->pts = nullptr;
    ev->d2 = nullptr;
    ev->pix_cap = 0;
    cudaError_t e;
    if ((e = cudaMalloc((void**)&ev->col, (size_t)npx * 2 * sizeof(int))) != cudaSuccess) return e;
    if ((e = cudaMalloc((void**)&ev->pts, (size_t)npx * sizeof(float4))) != cudaSuccess) return e;
    if ((e = cudaMalloc((void**)&ev->d2, (size_t)npx * sizeof(float))) != cudaSuccess) return e;
    ev->pix_cap = npx;
    return cudaSuccess;
}

// The sensor points (whole warps of every tile), tile records and tile map of a
// w x h image (its tile count is not bounded by the pixels of another shape).
cudaError_t grow_tiles(ftr_ctx* c, EvalScratch* ev, int64_t n) {
    if (ev->tiles && ev->tiles_cap >= n) return cudaSuccess;
    cudaStreamSynchronize(c->stream);
    void* t = nullptr;
    if (ev->tiles) cudaFree(ev->tiles);
    ev->tiles = nullptr;
    ev->tiles_cap = 0;
    cudaError_t e = cudaMalloc(&t, (size_t)n * (256 * sizeof(float4) + sizeof(PointTile) + sizeof(int)));
    if (e == cudaSuccess) {
        ev->tiles = t;
        ev->tiles_cap = n;
    }
    return e;
}

cudaError_t grow_part(ftr_ctx* c, EvalScratch* ev, int64_t n) {
    if (ev->part_cap >= n) return cudaSuccess;
    cudaStreamSynchronize(c->stream);
    return grow(&ev->part, &ev->part_cap, n);
}

}  // namespace

EvalScratch* eval_scratch(ftr_ctx* c) {
    if (c->ev) return c->ev;
    EvalScratch* ev = new EvalScratch();
    if (cudaMalloc((void**)&ev->cnt, kCounters * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMallocHost((void**)&ev->h_res, 32 * sizeof(double)) != cudaSuccess) {
        if (ev->cnt) cudaFree(ev->cnt);
        delete ev;
        return nullptr;
    }
    c->ev = ev;
    return ev;
}

void eval_free(ftr_ctx* c) {
    EvalScratch* ev = c->ev;
    if (!ev) return;
    if (ev->zkey) cudaFree(ev->zkey);
    if (ev->big) cudaFree(ev->big);
    if (ev->proj) cudaFree(ev->proj);
    if (ev->col) cudaFree(ev->col);
    if (ev->pts) cudaFree(ev->pts);
    if (ev->d2) cudaFree(ev->d2);
    if (ev->tiles) cudaFree(ev->tiles);
    if (ev->cnt) cudaFree(ev->cnt);
    if (ev->part) cudaFree(ev->part);
    if (ev->h_res) cudaFreeHost(ev->h_res);
    if (ev->img) cudaFree(ev->img);
    if (ev->mask) cudaFree(ev->mask);
    delete ev;
    c->ev = nullptr;
}

}  // namespace ftr

using namespace ftr;

int ftr_eval_geometry(ftr_ctx* c, const ftr_camera* cam, const float* rendered_depth, const float* sensor_depth,
                      float* cp_d2_out, ftr_geometry_eval* out) {
    if (!c) return FTR_EINVAL;
    if (!camera_ok(cam) || !out)
        return set_err(c, FTR_EINVAL, "ftr_eval_geometry: a camera (w, h in 1..16384, focal != 0) and out");
    if (!dev_ptr(rendered_depth) || !dev_ptr(sensor_depth) || (cp_d2_out && !dev_ptr(cp_d2_out)))
        return set_err(c, FTR_EINVAL, "ftr_eval_geometry: depth images must be device memory");
    EvalScratch* ev = eval_scratch(c);
    if (!ev) return set_err(c, FTR_ENOMEM, "ftr_eval_geometry: scratch");
    const int w = cam->w, h = cam->h;
    const int64_t npx = (int64_t)w * h;
    cudaError_t e;
    if ((e = grow_pixels(c, ev, npx)) != cudaSuccess) return cuda_fail(c, e, "ftr_eval_geometry: scratch");
    if ((e = grow_part(c, ev, 4 * kSumBlocks)) != cudaSuccess) return cuda_fail(c, e, "ftr_eval_geometry: scratch");
    cudaStream_t st = c->stream;
    float* d2 = cp_d2_out ? cp_d2_out : ev->d2;
    int* colG = ev->col;
    int* colR = ev->col + npx;
    float4* ptsR = ev->pts;
    const int tx = (w + kTile - 1) / kTile, ty = (h + kTile - 1) / kTile;
    if ((e = grow_tiles(c, ev, (int64_t)tx * ty)) != cudaSuccess)
        return cuda_fail(c, e, "ftr_eval_geometry: scratch");
    float4* ptsG = static_cast<float4*>(ev->tiles);
    PointTile* tiles = reinterpret_cast<PointTile*>(ptsG + 256 * (int64_t)tx * ty);
    int* tile_of = reinterpret_cast<int*>(tiles + (int64_t)tx * ty);
    if ((e = cudaMemsetAsync(ev->cnt, 0, kCounters * sizeof(unsigned long long), st)) != cudaSuccess)
        return cuda_fail(c, e, "ftr_eval_geometry");
    const int nseg = (h + 31) / 32;
    if (col_smem(h) > 48 * 1024 && (e = allow_col_smem(c->device)) != cudaSuccess)
        return cuda_fail(c, e, "ftr_eval_geometry: column masks");
    k_ev_cols<<<(w + 31) / 32, 32 * (nseg < 16 ? nseg : 16), col_smem(h), st>>>(rendered_depth, sensor_depth, w, h,
                                                                               nseg, colG, colR, ev->cnt);
    k_ev_rows<<<h, 256, 0, st>>>(rendered_depth, sensor_depth, w, colG, colR, ev->cnt);
    Intr in;
    for (int j = 0; j < 9; ++j) in.K[j] = cam->K[j];
    k_ev_points<<<dim3((unsigned)tx, (unsigned)ty), 256, 0, st>>>(rendered_depth, sensor_depth, w, h, in, ptsG, ptsR,
                                                                 tiles, tile_of, d2, ev->cnt);
    // the list sizes stay on the device: CTAs past the sensor points end at once
    k_ev_cp<<<(unsigned)((int64_t)tx * ty * (256 / kCpThreads)), kCpThreads, 0, st>>>(ptsG, ptsR, tiles, tile_of, w,
                                                                                          ev->cnt, d2);
    k_sum<float><<<kSumBlocks, 256, 0, st>>>(d2, npx, ev->part);
    k_sum_final<<<1, 256, 0, st>>>(ev->part, kSumBlocks, reinterpret_cast<double*>(ev->cnt + 9));
    c->launches += 6;
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(c, e, "ftr_eval_geometry: kernels");
    unsigned long long* hc = reinterpret_cast<unsigned long long*>(ev->h_res);
    if ((e = cudaMemcpyAsync(hc, ev->cnt, kCounters * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st)) !=
            cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return cuda_fail(c, e, "ftr_eval_geometry: results");
    const int64_t I = (int64_t)hc[6], J = (int64_t)hc[7];
    out->rendered_px = (int64_t)hc[0];
    out->sensor_px = (int64_t)hc[1];
    out->xor_px = (int64_t)hc[2];
    out->or_px = (int64_t)hc[3];
    out->vre = out->or_px ? (double)out->xor_px / (double)out->or_px : 0.0;
    const double inf = std::numeric_limits<double>::infinity();
    if (out->rendered_px == 0 && out->sensor_px == 0)
        out->hausdorff_px = 0.0;
    else if (out->rendered_px == 0 || out->sensor_px == 0)
        out->hausdorff_px = inf;
    else
        out->hausdorff_px = sqrt((double)(hc[4] > hc[5] ? hc[4] : hc[5]));
    out->sensor_points = I;
    out->rendered_points = J;
    if (I == 0)
        out->cp_rmse = std::numeric_limits<double>::quiet_NaN();
    else if (J == 0)
        out->cp_rmse = inf;
    else
        out->cp_rmse = sqrt(ev->h_res[9] / (double)I);
    return FTR_OK;
}

int ftr_eval_appearance(ftr_ctx* c, int w, int h, const float* rendered_depth, const uint8_t* rendered_rgb,
                        const uint8_t* sensor_rgb, ftr_appearance_eval* out) {
    if (!c) return FTR_EINVAL;
    if (w < 1 || h < 1 || w > 16384 || h > 16384 || !out)
        return set_err(c, FTR_EINVAL, "ftr_eval_appearance: 1 <= w, h <= 16384 and out");
    if (!dev_ptr(rendered_depth) || !dev_ptr(rendered_rgb) || !dev_ptr(sensor_rgb))
        return set_err(c, FTR_EINVAL, "ftr_eval_appearance: images must be device memory");
    EvalScratch* ev = eval_scratch(c);
    if (!ev) return set_err(c, FTR_ENOMEM, "ftr_eval_appearance: scratch");
    int ws[3], hs[3];
    int64_t off[4] = {0, 0, 0, 0}, boff[4] = {0, 0, 0, 0};
    unsigned gx[3], gy[3];
    for (int j = 0; j < 3; ++j) {
        ws[j] = j ? ws[j - 1] / 2 : w;
        hs[j] = j ? hs[j - 1] / 2 : h;
        off[j + 1] = off[j] + (int64_t)ws[j] * hs[j];
        gx[j] = (unsigned)((ws[j] + kSsimW - 1) / kSsimW);
        gy[j] = (unsigned)((hs[j] + kSsimH - 1) / kSsimH);
        boff[j + 1] = boff[j] + (int64_t)gx[j] * gy[j];
    }
    const double nan = std::numeric_limits<double>::quiet_NaN();
    cudaError_t e;
    const int64_t planes = off[3];
    if (planes > ev->img_cap) {
        cudaStreamSynchronize(c->stream);
        if (ev->img) cudaFree(ev->img);
        if (ev->mask) cudaFree(ev->mask);
        ev->img = nullptr;
        ev->mask = nullptr;
        ev->img_cap = 0;
        if ((e = cudaMalloc((void**)&ev->img, (size_t)planes * 2 * sizeof(float))) != cudaSuccess ||
            (e = cudaMalloc((void**)&ev->mask, (size_t)planes)) != cudaSuccess)
            return cuda_fail(c, e, "ftr_eval_appearance: scratch");
        ev->img_cap = planes;
    }
    if ((e = grow_part(c, ev, 4 * boff[3] + 16)) != cudaSuccess) return cuda_fail(c, e, "ftr_eval_appearance");
    cudaStream_t st = c->stream;
    float* X = ev->img;
    float* Y = ev->img + planes;
    uint8_t* S = ev->mask;
    k_ap_luma<<<(unsigned)((off[1] + 255) / 256), 256, 0, st>>>(rendered_rgb, sensor_rgb, rendered_depth, off[1], X,
                                                                 Y, S);
    c->launches++;
    Taps tp;
    for (int i = -kR; i <= kR; ++i) tp.g[i + kR] = (float)exp(-(double)(i * i) / (2.0 * 1.5 * 1.5));
    for (int j = 1; j < 3; ++j) {
        const int64_t n = (int64_t)ws[j] * hs[j];
        if (n > 0) {
            k_ap_down<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(X + off[j - 1], Y + off[j - 1], S + off[j - 1],
                                                                   ws[j - 1], ws[j], hs[j], X + off[j], Y + off[j],
                                                                   S + off[j]);
            c->launches++;
        }
    }
    ApScales sc;
    for (int j = 0; j < 3; ++j) {
        sc.at[j] = boff[j];
        sc.plane[j] = off[j];
        sc.w[j] = ws[j];
        sc.h[j] = hs[j];
        sc.gx[j] = (int)gx[j];
    }
    sc.at[3] = boff[3];
    k_ap_ssim<<<(unsigned)boff[3], 256, 0, st>>>(X, Y, S, sc, tp, ev->part);
    c->launches++;
    k_ap_final<<<12, 256, 0, st>>>(ev->part, sc, ev->part + 4 * boff[3]);
    c->launches++;
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(c, e, "ftr_eval_appearance: kernels");
    if ((e = cudaMemcpyAsync(ev->h_res, ev->part + 4 * boff[3], 12 * sizeof(double), cudaMemcpyDeviceToHost, st)) !=
            cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return cuda_fail(c, e, "ftr_eval_appearance: sums");
    double prod = 1.0;
    for (int j = 0; j < 3; ++j) {
        const double* r = ev->h_res + 4 * j;
        const bool empty = (int64_t)gx[j] * gy[j] == 0 || !(r[3] > 0.0);
        if (empty) {
            for (int m = 0; m < 3; ++m) out->l[m] = out->c[m] = out->s[m] = nan;
            out->wms3im = nan;
            return FTR_OK;
        }
        out->l[j] = r[0] / r[3];
        out->c[j] = r[1] / r[3];
        out->s[j] = r[2] / r[3];
        const double vals[3] = {out->l[j], out->c[j], out->s[j]};
        const double ex[3] = {kAlpha[j], kBeta[j], kGamma[j]};
        for (int m = 0; m < 3; ++m)
            if (ex[m] != 0.0) prod *= pow(vals[m] > 0.0 ? vals[m] : 0.0, ex[m]);
    }
    out->wms3im = prod;
    return FTR_OK;
}

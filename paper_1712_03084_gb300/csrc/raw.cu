// Raw reconstruction of oriented, weighted points from depth maps (Sec. III-A).
//
// Per depth view and foreground pixel u (D(u) > 0): the camera point
// x_c = ((u_x - c_x) / f_x D, (u_y - c_y) / f_y D, D); its world point
// X = R^T (x_c - t); its normal from the organised triangulation of the pixel
// grid (two triangles per 2 x 2 quad, (p00, p01, p10) and (p01, p11, p10); a
// triangle is kept iff its pixels are foreground, its largest corner depth
// difference is <= step + 3 noise z_max^2 and its area is not zero; its unit
// normal faces the camera; the pixel's normal is the normalised sum of the
// kept triangles that contain it); its confidence W = W1 W2 with
// W1 = max(<-x_c / |x_c|, N>, 0) and W2 the mean of the silhouette over a
// (2r+1)^2 window, zero outside the image.  A pixel gives a point iff it is
// foreground and lies on a kept triangle.  Points come out in row-major pixel
// order per view.
//
// A CTA takes 32 x 16 pixels, a warp two rows of 32: their depths with a border
// of one, then every triangle of their quads once, then each pixel's sum of its six.
// Triangle edges are formed from exact depth differences (x_b - x_a = ((u_b - u_a)
// D_b + (u_a - c_x) (D_b - D_a)) / f_x), so the float32 normals keep ~1e-7 relative
// accuracy.  Every discrete decision (the depth-step test, the orientation flip, a
// zero normal sum) is taken in float32, and a pixel with one inside a guard band of
// its threshold is redone in float64 with the float64 formula, operation by
// operation.
//
// Launches per call: count (two bit masks, a word per 32 pixels of a row: the
// silhouette and the pixels that give a point), one-CTA scan of the points per
// eight words, emit (W2 from the silhouette mask; the normals of the points once
// more, which is less than the memory to keep them; the compacted points, normals,
// weights and the per-pixel confidence map).
//
// Bound by the instructions of the triangles and by the float64 redo of single
// pixels (some 5 us of dependent operations), not by bytes.  Six 512 x 424 views of a
// body (1.3 M pixels, 62 k points): count 29 -> 14 us, emit 63 -> 15 us against a
// thread per pixel of a row segment that formed its six triangles itself in both
// passes and summed 21 rows of depth tests for every column.
#include <cuda_runtime.h>
#include <math.h>

#include "ftr_internal.h"

namespace ftr {

namespace {

constexpr int kRawT = 256;
constexpr int kTileW = 32, kTileH = 16;                       // pixels per CTA
constexpr int kQuadW = kTileW + 1, kQuadH = kTileH + 1;       // quads that touch them
constexpr int kGroup = 8;                                     // mask words per entry of the scan
constexpr int kRawMaxR = 16;        // largest W2 radius (a window row of 33 bits)

struct RawView {
    int w, h;
    float fx, fy, cx, cy;
    double fxd, fyd, cxd, cyd;
    float R[9], t[3];
    const float* depth;
    float* conf;                    // nullable: per-pixel W
    int words;                      // mask words per row
    int word_base;                  // first mask word of this view; rows follow each other
};
struct RawSet {
    int k;
    RawView v[kMaxViews];
};

// A tile's depths (zero outside the image), pixel rays and triangles.
struct RawTile {
    float4 tri[2][kQuadH * kQuadW]; // by family and quad: unit normal; w = 0 dropped, 1 kept, 2 undecided
    float depth[kTileH + 2][kTileW + 3];
    float x[kTileW + 2], y[kTileH + 2];   // (u - c_x) / f_x, (v - c_y) / f_y
    unsigned short list[2 * kQuadH * kQuadW];
    int listed;
};

// Triangle (a, b, c) given by pixel offsets; returns false when a decision is
// too close to call in float32 (the caller redoes the pixel in float64).
struct Corner {
    int du, dv;
};

// Float64 restatement of one triangle, operation by operation as the plain
// definition (no fused multiply-add): keep flag and unit camera-facing normal.
__device__ bool tri_f64(const RawView& V, int u0, int v0, const Corner (&cn)[3], double step, double noise,
                        double n_out[3]) {
    double P[3][3], Z[3];
    for (int k = 0; k < 3; ++k) {
        const int u = u0 + cn[k].du, v = v0 + cn[k].dv;
        const double D = (double)V.depth[(int64_t)v * V.w + u];
        Z[k] = D;
        P[k][0] = __dmul_rn(__ddiv_rn(__dsub_rn((double)u, V.cxd), V.fxd), D);
        P[k][1] = __dmul_rn(__ddiv_rn(__dsub_rn((double)v, V.cyd), V.fyd), D);
        P[k][2] = D;
    }
    if (!(Z[0] > 0.0 && Z[1] > 0.0 && Z[2] > 0.0)) return false;
    const double zmax = fmax(fmax(Z[0], Z[1]), Z[2]);
    const double dz = fmax(fmax(fabs(Z[0] - Z[1]), fabs(Z[1] - Z[2])), fabs(Z[0] - Z[2]));
    const double thr = __dadd_rn(step, __dmul_rn(__dmul_rn(__dmul_rn(3.0, noise), zmax), zmax));
    double e1[3], e2[3];
    for (int c = 0; c < 3; ++c) {
        e1[c] = __dsub_rn(P[1][c], P[0][c]);
        e2[c] = __dsub_rn(P[2][c], P[0][c]);
    }
    double n[3] = {__dsub_rn(__dmul_rn(e1[1], e2[2]), __dmul_rn(e1[2], e2[1])),
                   __dsub_rn(__dmul_rn(e1[2], e2[0]), __dmul_rn(e1[0], e2[2])),
                   __dsub_rn(__dmul_rn(e1[0], e2[1]), __dmul_rn(e1[1], e2[0]))};
    const double ln = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(n[0], n[0]), __dmul_rn(n[1], n[1])),
                                           __dmul_rn(n[2], n[2])));
    if (!(dz <= thr) || !(ln > 0.0)) return false;
    double dot = 0.0;
    for (int c = 0; c < 3; ++c) {
        n[c] = __ddiv_rn(n[c], ln);
        const double cen = __ddiv_rn(__dadd_rn(__dadd_rn(P[0][c], P[1][c]), P[2][c]), 3.0);
        dot = __dadd_rn(dot, __dmul_rn(n[c], cen));
    }
    const double s = dot > 0.0 ? -1.0 : 1.0;
    for (int c = 0; c < 3; ++c) n_out[c] = s * n[c];
    return true;
}

// The depth-step test of a triangle with corner depths Z: 0 dropped, 2 undecided,
// 1 to be formed.
__device__ __forceinline__ int tri_test(float z0, float z1, float z2, float step, float noise) {
    if (!(z0 > 0.f && z1 > 0.f && z2 > 0.f)) return 0;
    const float zmax = fmaxf(fmaxf(z0, z1), z2);
    const float dz = fmaxf(fmaxf(fabsf(z0 - z1), fabsf(z1 - z2)), fabsf(z0 - z2));
    const float thr = step + 3.f * noise * zmax * zmax;
    if (fabsf(dz - thr) <= 1e-5f * thr) return 2;
    return dz > thr ? 0 : 1;
}

// Float32 triangle of family fam of the quad (qx, qy) of the tile at (x0, y0) that
// passed the test.  The two guards compare squares first, with a tenth to spare:
// only a triangle near one takes the square roots of its edges or centroid.
__device__ __forceinline__ float4 tri_f32(const RawView& V, const RawTile& T, int x0, int y0, int fam, int qx, int qy) {
    const float4 undecided = make_float4(0.f, 0.f, 0.f, 2.f);
    // corners: family A (0, 0) (1, 0) (0, 1), family B (1, 0) (1, 1) (0, 1)
    const float Z[3] = {T.depth[qy][qx + fam], T.depth[qy + fam][qx + 1], T.depth[qy + 1][qx]};
    // edges from exact depth differences; the steps in u and v are 0, 1 or -1
    const float ua = (float)(x0 - 1 + qx + fam) - V.cx, va = (float)(y0 - 1 + qy) - V.cy;
    float e[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float du = (float)(k == 0 ? 1 - fam : -fam), dv = (float)(k == 0 ? fam : 1);
        const float dd = Z[k + 1] - Z[0];
        e[k][0] = fmaf(ua, dd, du * Z[k + 1]) / V.fx;
        e[k][1] = fmaf(va, dd, dv * Z[k + 1]) / V.fy;
        e[k][2] = dd;
    }
    const float n[3] = {e[0][1] * e[1][2] - e[0][2] * e[1][1], e[0][2] * e[1][0] - e[0][0] * e[1][2],
                        e[0][0] * e[1][1] - e[0][1] * e[1][0]};
    const float n2 = n[0] * n[0] + n[1] * n[1] + n[2] * n[2], ln = sqrtf(n2);
    const float a2 = e[0][0] * e[0][0] + e[0][1] * e[0][1] + e[0][2] * e[0][2];
    const float b2 = e[1][0] * e[1][0] + e[1][1] * e[1][1] + e[1][2] * e[1][2];
    if (!(n2 > 1.1e-10f * a2 * b2 && n2 > 1e-30f) && !(ln > 1e-5f * (sqrtf(a2) * sqrtf(b2))))
        return undecided;                         // (nearly) degenerate
    // orientation: n . centroid
    float cen[3] = {0.f, 0.f, 0.f};
    cen[0] += T.x[qx + fam] * Z[0];
    cen[0] += T.x[qx + 1] * Z[1];
    cen[0] += T.x[qx] * Z[2];
    cen[1] += T.y[qy] * Z[0];
    cen[1] += T.y[qy + fam] * Z[1];
    cen[1] += T.y[qy + 1] * Z[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) cen[2] += Z[k];
    const float dot = n[0] * cen[0] + n[1] * cen[1] + n[2] * cen[2];
    const float c2 = cen[0] * cen[0] + cen[1] * cen[1] + cen[2] * cen[2];
    if (!(dot * dot > 1.1e-8f * n2 * c2 && dot * dot > 1e-30f) && fabsf(dot) <= 1e-4f * ln * sqrtf(c2))
        return undecided;
    const float s = (dot > 0.f ? -1.f : 1.f) / ln;
    return make_float4(__fmul_rn(s, n[0]), __fmul_rn(s, n[1]), __fmul_rn(s, n[2]), 1.f);
}

// Depth of the image pixel, zero outside.
__device__ __forceinline__ float depth_at(const RawView& V, int u, int v) {
    return u >= 0 && v >= 0 && u < V.w && v < V.h ? V.depth[(int64_t)v * V.w + u] : 0.f;
}

// The depths of the tile's pixels; whether one is foreground.
__device__ __forceinline__ bool load_tile(RawTile& T, const RawView& V, int x0, int y0) {
    const int c = threadIdx.x % kTileW;
    bool fg = false;
#pragma unroll
    for (int k = 0; k < kTileW * kTileH / kRawT; ++k) {
        const int r = threadIdx.x / kTileW + k * (kRawT / kTileW);
        const float d = x0 + c < V.w && y0 + r < V.h ? V.depth[(int64_t)(y0 + r) * V.w + x0 + c] : 0.f;
        T.depth[r + 1][c + 1] = d;
        fg |= d > 0.f;
    }
    if (threadIdx.x == 0) T.listed = 0;
    return __syncthreads_or(fg);
}

// The border of the tile, its rays, and every triangle of its quads: the depth-step
// test by quads, then the triangles that passed it, listed so that warps are full
// (a body covers about a third of the tiles that it touches).
__device__ __forceinline__ void tile_triangles(RawTile& T, const RawView& V, int x0, int y0, float step, float noise) {
    constexpr int kQ = kQuadW * kQuadH, kRows = 2 * (kTileW + 2), kBorder = kRows + 2 * kTileH;
    static_assert(kBorder + kTileW + 2 + kTileH + 2 <= kRawT, "one thread per border pixel and ray");
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < kBorder) {
        const int e = tid - kRows;                     // the two rows, then the two columns
        const int r = tid < kRows ? (tid & 1) * (kTileH + 1) : 1 + (e >> 1);
        const int c = tid < kRows ? tid >> 1 : (e & 1) * (kTileW + 1);
        T.depth[r][c] = depth_at(V, x0 - 1 + c, y0 - 1 + r);
    } else if (tid < kBorder + kTileW + 2) {
        const int c = tid - kBorder;
        T.x[c] = ((float)(x0 - 1 + c) - V.cx) / V.fx;
    } else if (tid < kBorder + kTileW + 2 + kTileH + 2) {
        const int r = tid - kBorder - (kTileW + 2);
        T.y[r] = ((float)(y0 - 1 + r) - V.cy) / V.fy;
    }
    __syncthreads();
    for (int base = 0; base < kQ; base += kRawT) {
        const int q = base + tid, qy = q / kQuadW, qx = q - qy * kQuadW;
        int st[2] = {0, 0};
        if (q < kQ) {
            const float z00 = T.depth[qy][qx], z10 = T.depth[qy][qx + 1], z01 = T.depth[qy + 1][qx],
                        z11 = T.depth[qy + 1][qx + 1];
            st[0] = tri_test(z00, z10, z01, step, noise);
            st[1] = tri_test(z10, z11, z01, step, noise);
        }
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const unsigned m = __ballot_sync(0xffffffffu, st[f] == 1);
            int at = 0;
            if (m && lane == 0) at = atomicAdd(&T.listed, __popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (st[f] == 1) T.list[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)(f * kQ + q);
            else if (q < kQ) T.tri[f][q] = make_float4(0.f, 0.f, 0.f, (float)st[f]);
        }
    }
    __syncthreads();
    for (int k = tid; k < T.listed; k += kRawT) {
        const int i = T.list[k], fam = i >= kQ, q = i - fam * kQ, qy = q / kQuadW;
        T.tri[fam][q] = tri_f32(V, T, x0, y0, fam, q - qy * kQuadW, qy);
    }
    __syncthreads();
}

// The six triangles containing pixel (u, v): (quad offset, family).
__device__ __forceinline__ void tri_of(int t, int& qu, int& qv, Corner (&cn)[3]) {
    // family A: (0,0) (1,0) (0,1) in (du, dv); family B: (1,0) (1,1) (0,1)
    const int fam = t < 3 ? 0 : 1;
    if (fam == 0) {
        cn[0] = {0, 0};
        cn[1] = {1, 0};
        cn[2] = {0, 1};
    } else {
        cn[0] = {1, 0};
        cn[1] = {1, 1};
        cn[2] = {0, 1};
    }
    // quads whose family-A triangle contains the pixel: (0,0) (-1,0) (0,-1);
    // family B: (-1,0) (-1,-1) (0,-1)
    const int qa[3][2] = {{0, 0}, {-1, 0}, {0, -1}};
    const int qb[3][2] = {{-1, 0}, {-1, -1}, {0, -1}};
    qu = fam == 0 ? qa[t][0] : qb[t - 3][0];
    qv = fam == 0 ? qa[t][1] : qb[t - 3][1];
}

// Camera-space unit normal of pixel (c, r) of the tile, image pixel (u, v); 1 =
// a point, 0 = none or not asked for.  All lanes of the warp take part: the pixels
// that float32 leaves open are redone in float64, four at a time with a lane per
// triangle (the float64 unit takes as long for one lane as for all).
__device__ __forceinline__ int pixel_normal(const RawView& V, const RawTile& T, int c0, int r, int u, int v, bool ask,
                                            double stepd, double noised, float n[3]) {
    const int lane = threadIdx.x & 31;
    int p = 0;
    if (ask) {
        const int q = r * kQuadW + c0;                 // quad (u - 1, v - 1)
        const float4 t[6] = {T.tri[0][q + kQuadW + 1], T.tri[0][q + kQuadW], T.tri[0][q + 1],
                             T.tri[1][q + kQuadW],     T.tri[1][q],          T.tri[1][q + 1]};
        float acc[3] = {0.f, 0.f, 0.f}, state = 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) {                  // a dropped one adds zeros
            acc[0] += t[k].x;
            acc[1] += t[k].y;
            acc[2] += t[k].z;
            state = fmaxf(state, t[k].w);
        }
        const float l2 = acc[0] * acc[0] + acc[1] * acc[1] + acc[2] * acc[2];
        if (state == 1.f && l2 > 1e-6f) {
            const float inv = rsqrtf(l2);
            for (int c = 0; c < 3; ++c) n[c] = acc[c] * inv;
            p = 1;
        } else if (state > 0.f) {                      // undecided, or the unit normals (nearly) cancel
            p = -1;
        }
    }
    for (unsigned open = __ballot_sync(0xffffffffu, p < 0); open;) {
        // the pixel of this lane's group of eight, and the group of this lane's pixel
        unsigned rest = open;
        int src = -1, mine = -1;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int l = __ffs(rest) - 1;         // -1: none left
            if (l >= 0) {
                if (g == lane >> 3) src = l;
                if (l == lane) mine = g;
                rest &= rest - 1u;
            }
        }
        open = rest;
        const int us = __shfl_sync(0xffffffffu, u, src < 0 ? 0 : src);
        const int vs = __shfl_sync(0xffffffffu, v, src < 0 ? 0 : src);
        const int t = lane & 7;
        double tn[3] = {0.0, 0.0, 0.0};
        bool keep = false;
        if (src >= 0 && t < 6) {
            int qu, qv;
            Corner cn[3];
            tri_of(t, qu, qv, cn);
            const int u0 = us + qu, v0 = vs + qv;
            if (u0 >= 0 && v0 >= 0 && u0 < V.w - 1 && v0 < V.h - 1) keep = tri_f64(V, u0, v0, cn, stepd, noised, tn);
        }
        const unsigned kept = __ballot_sync(0xffffffffu, keep);
        double a[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int from = 8 * (mine < 0 ? 0 : mine) + k;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double x = __shfl_sync(0xffffffffu, tn[c], from);
                if (kept >> from & 1u) a[c] = __dadd_rn(a[c], x);
            }
        }
        if (mine >= 0) {
            const double ln = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
            p = ln > 0.0;
            if (p)
                for (int c = 0; c < 3; ++c) n[c] = (float)(a[c] / ln);
        }
    }
    return p;
}

// The masks: bit i of word k of a row = pixel 32 k + i (zero past the image).
__global__ void __launch_bounds__(kRawT) k_raw_count(const __grid_constant__ RawSet S, float step, float noise,
                                                     double stepd, double noised, unsigned* __restrict__ sil,
                                                     unsigned* __restrict__ val) {
    pdl_wait();
    __shared__ RawTile T;
    const RawView& V = S.v[blockIdx.z];
    const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kTileH;
    if (x0 >= V.w || y0 >= V.h) return;            // block-uniform
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool fg = load_tile(T, V, x0, y0);
    if (fg) tile_triangles(T, V, x0, y0, step, noise);
    for (int r = wid; r < kTileH; r += kRawT / 32) {
        const int v = y0 + r;
        if (v >= V.h) break;                       // warp-uniform
        unsigned bs = 0u, bv = 0u;
        if (fg) {
            const bool in = T.depth[r + 1][lane + 1] > 0.f;
            float n[3];
            const int p = pixel_normal(V, T, lane, r, x0 + lane, v, in, stepd, noised, n);
            bs = __ballot_sync(0xffffffffu, in);
            bv = __ballot_sync(0xffffffffu, p != 0);
        }
        if (lane == 0) {
            const int at = V.word_base + v * V.words + blockIdx.x;
            sil[at] = bs;
            val[at] = bv;
        }
    }
}

// One CTA: off[g] = the points before group g of kGroup mask words; all of them
// into *total.  Four groups per thread and round, a thousand apart.
__global__ void __launch_bounds__(1024) k_raw_scan(const unsigned* __restrict__ val, int words,
                                                   int* __restrict__ off, int* total) {
    pdl_wait();
    constexpr int kPer = 4;
    __shared__ int sh[kPer * 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int groups = (words + kGroup - 1) / kGroup;
    int carry = 0;
    for (int base = 0; base < groups; base += kPer * 1024) {
        int c[kPer], inc[kPer];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int g = base + k * 1024 + threadIdx.x;
            c[k] = 0;
            if ((g + 1) * kGroup <= words) {
                const uint4* q = reinterpret_cast<const uint4*>(val + g * kGroup);
                const uint4 a = q[0], b = q[1];
                c[k] = __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w) + __popc(b.x) + __popc(b.y) +
                       __popc(b.z) + __popc(b.w);
            } else {
                for (int i = g * kGroup; i < words; ++i) c[k] += __popc(val[i]);
            }
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) inc[k] = c[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int x = __shfl_up_sync(0xffffffffu, inc[k], o);
                if (lane >= o) inc[k] += x;
            }
        if (lane == 31)
#pragma unroll
            for (int k = 0; k < kPer; ++k) sh[k * 32 + wid] = inc[k];
        __syncthreads();
        if (wid == 0) {                                // the 128 warp sums, four per lane
            int w[kPer], sum = 0;
#pragma unroll
            for (int k = 0; k < kPer; ++k) sum += w[k] = sh[lane * kPer + k];
            int x = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            x -= sum;
#pragma unroll
            for (int k = 0; k < kPer; ++k) sh[lane * kPer + k] = x += w[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int g = base + k * 1024 + threadIdx.x, at = k * 32 + wid;
            if (g < groups) off[g] = carry + (at ? sh[at - 1] : 0) + inc[k] - c[k];
        }
        carry += sh[kPer * 32 - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// The tile's points are listed first, so that warps are full; the others only get
// their zero in the confidence map.  W2 counts the silhouette bits of the window,
// two mask words per window row.
__global__ void __launch_bounds__(kRawT) k_raw_emit(const __grid_constant__ RawSet S, float step, float noise,
                                                    double stepd, double noised, int radius,
                                                    const int* __restrict__ off, const unsigned* __restrict__ sil,
                                                    const unsigned* __restrict__ val, float* __restrict__ P,
                                                    float* __restrict__ N, float* __restrict__ W) {
    pdl_wait();
    constexpr int kRows = kTileH + 2 * kRawMaxR;
    __shared__ RawTile T;
    __shared__ unsigned win[kRows][3];                 // silhouette words of the windows' rows
    __shared__ int slot0[kTileH], before[kTileH + 1];  // by row: its first point's slot; points of the rows before
    __shared__ unsigned short pts[kTileW * kTileH];
    const RawView& V = S.v[blockIdx.z];
    const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kTileH;
    if (x0 >= V.w || y0 >= V.h) return;                // block-uniform
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int first = V.word_base + y0 * V.words + blockIdx.x;
    const int row = min(lane, kTileH - 1);             // lanes of each warp: the tile's rows
    const unsigned mine = lane < kTileH && y0 + row < V.h ? val[first + row * V.words] : 0u;
    const bool any = __any_sync(0xffffffffu, mine != 0u);   // the same in every warp
    if (V.conf)
        for (int r = wid; r < kTileH && y0 + r < V.h; r += kRawT / 32) {
            const unsigned bv = __shfl_sync(0xffffffffu, mine, r);
            if (x0 + lane < V.w && !(bv >> lane & 1u)) V.conf[(int64_t)(y0 + r) * V.w + x0 + lane] = 0.f;
        }
    if (!any) return;
    load_tile(T, V, x0, y0);
    if (wid == 0) {
        int inc = __popc(mine);
#pragma unroll
        for (int o = 1; o < kTileH; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += x;
        }
        if (lane < kTileH) {
            before[lane + 1] = inc;
            // points before the row's first one: of the groups before its word, the words before
            const int word = first + row * V.words;
            int at = 0;
            if (mine) {
                at = off[word / kGroup];
                for (int k = word / kGroup * kGroup; k < word; ++k) at += __popc(val[k]);
            }
            slot0[lane] = at;
        }
        if (lane == 0) before[0] = 0;
    }
    for (int i = tid; i < 3 * (kTileH + 2 * radius); i += kRawT) {
        const int r = i / 3, k = i - 3 * r, y = y0 - radius + r, w = blockIdx.x - 1 + k;
        win[r][k] = y >= 0 && y < V.h && w >= 0 && w < V.words ? sil[V.word_base + y * V.words + w] : 0u;
    }
    tile_triangles(T, V, x0, y0, step, noise);
    for (int r = wid; r < kTileH; r += kRawT / 32) {
        const unsigned bv = __shfl_sync(0xffffffffu, mine, r);
        if (bv >> lane & 1u) pts[before[r] + __popc(bv & ((1u << lane) - 1u))] = (unsigned short)(r * kTileW + lane);
    }
    __syncthreads();
    const int total = before[kTileH];
    for (int base = wid * 32; base < total; base += kRawT) {
        const bool ask = base + lane < total;
        const int id = ask ? pts[base + lane] : 0, r = id / kTileW, c = id % kTileW, u = x0 + c, v = y0 + r;
        float n[3];
        pixel_normal(V, T, c, r, u, v, ask, stepd, noised, n);
        if (!ask) continue;
        const int slot = slot0[r] + base + lane - before[r];
        // silhouette pixels u - radius .. u + radius of each window row: at most 33 bits
        // from bit (c - radius) mod 32 of its word, so two words hold them
        const int b0 = c - radius, w0 = 1 + (b0 >> 5), sh = b0 & 31;
        const unsigned long long window = (1ull << (2 * radius + 1)) - 1ull;
        int cnt = 0;
#pragma unroll 4
        for (int y = r; y <= r + 2 * radius; ++y) {
            const unsigned lo = win[y][w0], hi = win[y][w0 + 1];
            cnt += __popcll(((((unsigned long long)hi << 32) | lo) >> sh) & window);
        }
        const float k2 = (float)((2 * radius + 1) * (2 * radius + 1));
        const float D = T.depth[r + 1][c + 1];
        const float xc[3] = {T.x[c + 1] * D, T.y[r + 1] * D, D};
        const float l = sqrtf(xc[0] * xc[0] + xc[1] * xc[1] + xc[2] * xc[2]);
        const float w1 = fmaxf(-(xc[0] * n[0] + xc[1] * n[1] + xc[2] * n[2]) / l, 0.f);
        const float wk = w1 * ((float)cnt / k2);
        // world: R^T (x_c - t), R^T n
        const float d[3] = {xc[0] - V.t[0], xc[1] - V.t[1], xc[2] - V.t[2]};
        for (int k = 0; k < 3; ++k) {
            P[3 * (int64_t)slot + k] = V.R[k] * d[0] + V.R[3 + k] * d[1] + V.R[6 + k] * d[2];
            N[3 * (int64_t)slot + k] = V.R[k] * n[0] + V.R[3 + k] * n[1] + V.R[6 + k] * n[2];
        }
        W[slot] = wk;
        if (V.conf) V.conf[(int64_t)v * V.w + u] = wk;
    }
}

}  // namespace

cudaError_t launch_raw(ftr_ctx* c, const RawParams& rp, const ftr_view* views, int k, float* const* conf_maps,
                       float* P, float* N, float* W, int* scratch, int* d_total) {
    RawSet S{};
    S.k = k;
    int words = 0, max_tx = 0, max_ty = 0;
    for (int i = 0; i < k; ++i) {
        RawView& V = S.v[i];
        const ftr_view& src = views[i];
        V.w = src.w;
        V.h = src.h;
        V.fx = src.K[0];
        V.fy = src.K[4];
        V.cx = src.K[2];
        V.cy = src.K[5];
        V.fxd = src.K[0];
        V.fyd = src.K[4];
        V.cxd = src.K[2];
        V.cyd = src.K[5];
        for (int r = 0; r < 3; ++r) {
            for (int q = 0; q < 3; ++q) V.R[3 * r + q] = src.world_to_cam[4 * r + q];
            V.t[r] = src.world_to_cam[4 * r + 3];
        }
        V.depth = src.depth;
        V.conf = conf_maps ? conf_maps[i] : nullptr;
        V.words = (src.w + kTileW - 1) / kTileW;
        V.word_base = words;
        words += V.words * src.h;
        max_tx = max_tx > V.words ? max_tx : V.words;
        const int ty = (src.h + kTileH - 1) / kTileH;
        max_ty = max_ty > ty ? max_ty : ty;
    }
    const dim3 grid(max_tx, max_ty, k);
    // the point mask (its groups 32-byte aligned), the silhouette mask, the offsets of the groups
    unsigned* val = reinterpret_cast<unsigned*>(scratch);
    unsigned* sil = val + words;
    int* off = scratch + 2 * (int64_t)words;
    launch_pdl(k_raw_count, grid, kRawT, 0, c->stream, S, rp.step_f, rp.noise_f, rp.step, rp.noise, sil, val);
    launch_pdl(k_raw_scan, 1, 1024, 0, c->stream, (const unsigned*)val, words, off, d_total);
    launch_pdl(k_raw_emit, grid, kRawT, 0, c->stream, S, rp.step_f, rp.noise_f, rp.step, rp.noise, rp.radius,
               (const int*)off, (const unsigned*)sil, (const unsigned*)val, P, N, W);
    c->launches += 3;
    return cudaGetLastError();
}

int raw_scratch_ints(const ftr_view* views, int k) {
    int words = 0;
    for (int i = 0; i < k; ++i) words += ((views[i].w + kTileW - 1) / kTileW) * views[i].h;
    return 2 * words + (words + kGroup - 1) / kGroup;
}

int raw_max_radius() { return kRawMaxR; }

}  // namespace ftr

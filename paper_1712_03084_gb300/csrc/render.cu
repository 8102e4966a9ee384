// Rendering a triangle mesh into a pinhole camera (Sec. III-C, III-E).
//
// Sec. III-E projects the reconstructed mesh into every sensor view and reads
// back the depth and colour buffers; Sec. III-C draws each triangle with the
// per-vertex weights and UVs (multitexture blend).  No graphics API is used:
//
//   k_project  one thread per vertex: its camera coordinates in float64 and
//              its projection to 1e-7 pixels; the ray slopes of every pixel
//              column and row (float64);
//   k_raster   128 triangles per CTA: walk the pixel centres of the screen
//              bounding box, test coverage with the three edge functions,
//              intersect the pixel's ray with the triangle's plane and keep
//              the nearest surface with a 64-bit atomicMin on (float32 z bits
//              << 32 | triangle index); a triangle with more than 1024 pixel
//              centres in its box is listed instead and k_raster_big shares
//              its pixels among the threads of a CTA;
//   k_resolve  one thread per pixel: depth from the key, colour from the
//              winning triangle (perspective-correct barycentrics of the hit
//              point; vertex colours or the weighted blend of the views).
//
// Coverage and depth decide which triangle a pixel shows, so they are
// evaluated in float64 with every product, sum and quotient rounded on its
// own (no contraction) in one fixed order:
//   x_c = ((r0 X + r1 Y) + r2 Z) + t per row, a = x_c/z_c, b = y_c/z_c,
//   u = (K00 a + K01 b) + K02, v = K11 b + K12,
//   e_ab = (ub - ua)(py - va) - (vb - va)(px - ua) (and cyclic),
//   dy = (py - K12)/K11, dx = ((px - K02) - K01 dy)/K00,
//   n = (B - A) x (C - A), z = ((nx Ax + ny Ay) + nz Az) / ((nx dx + ny dy) + nz).
// float64 runs at 1/64 of the float32 rate, so k_raster takes a decision in
// float32 wherever its error bound allows and in float64 only where it does not
// (an edge function within its bound of zero), and the float64 work left (a
// depth per covered pixel that is not behind the surface already there) is
// queued per CTA so that it runs on full warps.  A triangle projected more
// than 2^20 pixels away, or not to a number, takes the float64 path throughout,
// and so do all triangles where the vertices cannot be projected ahead (see ftr_render).
// The colours are float32 (they only feed the final rounding to u8).
#include <cuda_runtime.h>
#include <math.h>

#include "ftr_internal.h"

namespace ftr {

namespace {

constexpr double kZNear = 0.01;     // metres: a triangle with a vertex nearer the camera plane is not drawn
constexpr int kBigPx = 1024;        // bounding-box pixels above which a triangle is shared by a CTA

struct CamDev {
    int w, h;
    double K[9], RT[12];
    float Kf[9], RTf[12];
};

struct TexDev {
    int k;
    int rgb_w[kMaxViews], rgb_h[kMaxViews];
    const uint8_t* rgb[kMaxViews];
};

__device__ __forceinline__ double dm(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double da(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double ds(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dd(double a, double b) { return __ddiv_rn(a, b); }

__device__ __forceinline__ void cam_point(const CamDev& c, const float* X, double xc[3]) {
    const double x = X[0], y = X[1], z = X[2];
#pragma unroll
    for (int r = 0; r < 3; ++r)
        xc[r] = da(da(da(dm(c.RT[4 * r], x), dm(c.RT[4 * r + 1], y)), dm(c.RT[4 * r + 2], z)), c.RT[4 * r + 3]);
}

__device__ __forceinline__ double edge(double ua, double va, double ub, double vb, double px, double py) {
    return ds(dm(ds(ub, ua), ds(py, va)), dm(ds(vb, va), ds(px, ua)));
}

// Everything a pixel test needs, set up once per triangle.
struct TriSetup {
    double u[3], v[3];
    double nx, ny, nz, num;
    double x0, x1, y0, y1;
};

// Projects the triangle and its plane; false if it is not drawn (an index
// out of range, a vertex nearer than kZNear, zero area, or no pixel centre
// in its clipped bounding box).
__device__ __forceinline__ bool tri_setup(const CamDev& cam, const float* __restrict__ verts,
                                          const int32_t* __restrict__ tris, int64_t t, int64_t nv, TriSetup& s) {
    const int i3[3] = {tris[3 * t], tris[3 * t + 1], tris[3 * t + 2]};
    double xc[3][3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        if (i3[m] < 0 || i3[m] >= nv) return false;
        cam_point(cam, verts + 3 * (int64_t)i3[m], xc[m]);
        if (!(xc[m][2] >= kZNear)) return false;
        const double a = dd(xc[m][0], xc[m][2]);
        const double b = dd(xc[m][1], xc[m][2]);
        s.u[m] = da(da(dm(cam.K[0], a), dm(cam.K[1], b)), cam.K[2]);
        s.v[m] = da(dm(cam.K[4], b), cam.K[5]);
    }
    const double area = ds(dm(ds(s.u[1], s.u[0]), ds(s.v[2], s.v[0])), dm(ds(s.v[1], s.v[0]), ds(s.u[2], s.u[0])));
    if (!isfinite(area) || area == 0.0) return false;
    s.x0 = fmax(ceil(fmin(fmin(s.u[0], s.u[1]), s.u[2])), 0.0);
    s.x1 = fmin(floor(fmax(fmax(s.u[0], s.u[1]), s.u[2])), (double)(cam.w - 1));
    s.y0 = fmax(ceil(fmin(fmin(s.v[0], s.v[1]), s.v[2])), 0.0);
    s.y1 = fmin(floor(fmax(fmax(s.v[0], s.v[1]), s.v[2])), (double)(cam.h - 1));
    if (s.x1 < s.x0 || s.y1 < s.y0) return false;
    double e1v[3], e2v[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        e1v[r] = ds(xc[1][r], xc[0][r]);
        e2v[r] = ds(xc[2][r], xc[0][r]);
    }
    s.nx = ds(dm(e1v[1], e2v[2]), dm(e1v[2], e2v[1]));
    s.ny = ds(dm(e1v[2], e2v[0]), dm(e1v[0], e2v[2]));
    s.nz = ds(dm(e1v[0], e2v[1]), dm(e1v[1], e2v[0]));
    s.num = da(da(dm(s.nx, xc[0][0]), dm(s.ny, xc[0][1])), dm(s.nz, xc[0][2]));
    return true;
}

// Coverage and depth of pixel (px, py) (dy = its ray's y slope); the key
// goes to the z-buffer when the pixel is covered.
__device__ __forceinline__ void tri_pixel(const CamDev& cam, const TriSetup& s, double px, double py, double dy,
                                          unsigned long long tid, unsigned long long* __restrict__ zkey) {
    const double e0 = edge(s.u[0], s.v[0], s.u[1], s.v[1], px, py);
    const double e1 = edge(s.u[1], s.v[1], s.u[2], s.v[2], px, py);
    const double e2 = edge(s.u[2], s.v[2], s.u[0], s.v[0], px, py);
    const bool in = (e0 >= 0.0 && e1 >= 0.0 && e2 >= 0.0) || (e0 <= 0.0 && e1 <= 0.0 && e2 <= 0.0);
    if (!in) return;
    const double dx = dd(ds(ds(px, cam.K[2]), dm(cam.K[1], dy)), cam.K[0]);
    const double den = da(da(dm(s.nx, dx), dm(s.ny, dy)), s.nz);
    if (den == 0.0) return;
    const double z = dd(s.num, den);
    if (!(z > 0.0) || !isfinite(z)) return;
    const unsigned long long key = ((unsigned long long)__float_as_uint(__double2float_rn(z)) << 32) | tid;
    atomicMin(zkey + (int64_t)py * cam.w + (int64_t)px, key);
}

// Per vertex: at = the projection rounded to whole pixels (int bits) and the
// rest in float32; xyz = camera coordinates in float32 and how to treat the
// vertex; vd = the camera coordinates in float64.
//
// The rest is good to 1e-7 pixels at any image position, so that few coverage
// decisions are left open: x / z = a + da with a the float32 quotient and da
// from the exact remainder x - a z (one float64 operation), and every product
// and sum that follows keeps its float32 rounding error as a second term.
// (Plain float32 projections, 1e-3 pixels, left one fragment in sixteen open
// and with it a float64 coverage test in every warp: 97 us instead of 32 for
// the 1920 x 1080 raster below.)
constexpr float kVertSkip = -1.f, kVertExact = 0.f, kVertFast = 1.f;

__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

__device__ __forceinline__ float two_prod(float a, float b, float& err) {
    const float p = __fmul_rn(a, b);
    err = __fmaf_rn(a, b, -p);
    return p;
}

__global__ void __launch_bounds__(256) k_project(CamDev cam, const float* __restrict__ verts, int64_t nv,
                                                 float4* __restrict__ at, float4* __restrict__ xyz,
                                                 double* __restrict__ vd, double* __restrict__ slope) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nv) {
        double xc[3];
        cam_point(cam, verts + 3 * i, xc);
#pragma unroll
        for (int r = 0; r < 3; ++r) vd[3 * i + r] = xc[r];
        const float x = (float)xc[0], y = (float)xc[1], z = (float)xc[2];
        const float a = x / z, b = y / z;
        const float ar = (float)__fma_rn(-(double)a, xc[2], xc[0]) / z, br = (float)__fma_rn(-(double)b, xc[2], xc[1]) / z;
        float e1, e2, e3, e4, e5, e6;
        const float ua = two_prod(cam.Kf[0], a, e1), ub = two_prod(cam.Kf[1], b, e2);
        const float us = two_sum(two_sum(ua, ub, e3), cam.Kf[2], e4);
        const float ul = ((e1 + e2) + (e3 + e4)) + (cam.Kf[0] * ar + cam.Kf[1] * br);
        const float va = two_prod(cam.Kf[4], b, e5), vs = two_sum(va, cam.Kf[5], e6);
        const float vl = (e5 + e6) + cam.Kf[4] * br;
        const float ui = rintf(us), vi = rintf(vs);
        // the second terms are below 2^-23 of the sums they belong to, their own
        // errors below 2^-45 of them (2^-25 pixels at the limit of 2^20), and the rest
        // (half a pixel and a second term) rounds by 2^-25: 6e-8 together
        const float size = fabsf(ua) + fabsf(ub) + fabsf(cam.Kf[2]) + fabsf(va) + fabsf(cam.Kf[5]);
        const float how = !(xc[2] >= kZNear) ? kVertSkip : (size < 1048576.f ? kVertFast : kVertExact);
        at[i] = make_float4(__int_as_float((int)ui), __int_as_float((int)vi), (us - ui) + ul, (vs - vi) + vl);
        xyz[i] = make_float4(x, y, z, how);
    } else {
        // slope[x] = (x - K02) / K00 (rays without skew), slope[w + y] = (y - K12) / K11
        const int64_t k = i - nv;
        if (k < cam.w)
            slope[k] = dd(ds((double)k, cam.K[2]), cam.K[0]);
        else if (k < cam.w + cam.h)
            slope[k] = dd(ds((double)(k - cam.w), cam.K[5]), cam.K[4]);
    }
}

constexpr int kRasterThreads = 128;

// The float64 path of one triangle throughout.
__device__ __noinline__ void raster_exact(const CamDev& cam, const float* __restrict__ verts,
                                          const int32_t* __restrict__ tris, int64_t t, int64_t nv,
                                          unsigned long long* __restrict__ zkey, int* __restrict__ big,
                                          int* __restrict__ nbig) {
    TriSetup s;
    if (!tri_setup(cam, verts, tris, t, nv, s)) return;
    if ((s.x1 - s.x0 + 1.0) * (s.y1 - s.y0 + 1.0) > (double)kBigPx) {
        big[atomicAdd(nbig, 1)] = (int)t;          // at most nt entries
        return;
    }
    for (double py = s.y0; py <= s.y1; py += 1.0) {
        const double dy = dd(ds(py, cam.K[5]), cam.K[4]);
        for (double px = s.x0; px <= s.x1; px += 1.0) tri_pixel(cam, s, px, py, dy, (unsigned long long)t, zkey);
    }
}

// All triangles that way: nothing is projected ahead.
__global__ void __launch_bounds__(kRasterThreads) k_raster_exact(CamDev cam, const float* __restrict__ verts,
                                                                 const int32_t* __restrict__ tris, int64_t nt,
                                                                 int64_t nv, unsigned long long* __restrict__ zkey,
                                                                 int* __restrict__ big, int* __restrict__ nbig) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nt) raster_exact(cam, verts, tris, t, nv, zkey, big, nbig);
}

// Coverage of pixel (px, py) in float64, for a pixel whose float32 edge
// functions leave it open: projections, area, bounding box and edges as in
// tri_setup and tri_pixel.
__device__ __noinline__ bool covered_exact(const CamDev& cam, const double* __restrict__ vd, int i0, int i1, int i2,
                                           int pxi, int pyi) {
    const int id[3] = {i0, i1, i2};
    double u[3], v[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const double* xc = vd + 3 * (int64_t)id[m];
        const double a = dd(xc[0], xc[2]), b = dd(xc[1], xc[2]);
        u[m] = da(da(dm(cam.K[0], a), dm(cam.K[1], b)), cam.K[2]);
        v[m] = da(dm(cam.K[4], b), cam.K[5]);
    }
    const double area = ds(dm(ds(u[1], u[0]), ds(v[2], v[0])), dm(ds(v[1], v[0]), ds(u[2], u[0])));
    if (!isfinite(area) || area == 0.0) return false;
    const double px = pxi, py = pyi;
    if (px < fmin(fmin(u[0], u[1]), u[2]) || px > fmax(fmax(u[0], u[1]), u[2]) ||
        py < fmin(fmin(v[0], v[1]), v[2]) || py > fmax(fmax(v[0], v[1]), v[2]))
        return false;
    const double e0 = edge(u[0], v[0], u[1], v[1], px, py);
    const double e1 = edge(u[1], v[1], u[2], v[2], px, py);
    const double e2 = edge(u[2], v[2], u[0], v[0], px, py);
    return (e0 >= 0.0 && e1 >= 0.0 && e2 >= 0.0) || (e0 <= 0.0 && e1 <= 0.0 && e2 <= 0.0);
}

// Plane of a triangle in float64 (n, n . A), as in tri_setup.
__device__ __forceinline__ void plane_exact(const double* __restrict__ vd, int i0, int i1, int i2, double out[4]) {
    double A[3], e1v[3], e2v[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        A[r] = vd[3 * (int64_t)i0 + r];
        e1v[r] = ds(vd[3 * (int64_t)i1 + r], A[r]);
        e2v[r] = ds(vd[3 * (int64_t)i2 + r], A[r]);
    }
    out[0] = ds(dm(e1v[1], e2v[2]), dm(e1v[2], e2v[1]));
    out[1] = ds(dm(e1v[2], e2v[0]), dm(e1v[0], e2v[2]));
    out[2] = ds(dm(e1v[0], e2v[1]), dm(e1v[1], e2v[0]));
    out[3] = da(da(dm(out[0], A[0]), dm(out[1], A[1])), dm(out[2], A[2]));
}

// Depth of a covered pixel and its z-buffer entry, as in tri_pixel; slope holds
// the same quotients (with skew the x slope depends on y and is formed here).
__device__ __forceinline__ void depth_exact(const CamDev& cam, const double n[4], int px, int py,
                                            const double* __restrict__ slope, unsigned long long t,
                                            unsigned long long* __restrict__ zkey) {
    const double dy = slope[cam.w + py];
    const double dx = cam.K[1] == 0.0 ? slope[px]
                                      : dd(ds(ds((double)px, cam.K[2]), dm(cam.K[1], dy)), cam.K[0]);
    const double den = da(da(dm(n[0], dx), dm(n[1], dy)), n[2]);
    if (den == 0.0) return;
    const double z = dd(n[3], den);
    if (!(z > 0.0) || !isfinite(z)) return;
    const unsigned long long key = ((unsigned long long)__float_as_uint(__double2float_rn(z)) << 32) | t;
    atomicMin(zkey + (int64_t)py * cam.w + px, key);
}

constexpr int kQueue = 2048;        // fragments per CTA that wait for their float64 depth (8 KB)

// Measured on 152,000 triangles of a body-sized mesh: 88 us at 512 x 424 and
// 213 us at 1920 x 1080 with one float64 thread per triangle and pixel walk,
// 18 and 32 us now.
__global__ void __launch_bounds__(kRasterThreads) k_raster(
    CamDev cam, const float* __restrict__ verts, const int32_t* __restrict__ tris, int64_t nt, int64_t nv,
    const float4* __restrict__ at, const float4* __restrict__ xyz, const double* __restrict__ vd,
    const double* __restrict__ slope, unsigned long long* __restrict__ zkey, int* __restrict__ big,
    int* __restrict__ nbig) {
    __shared__ unsigned s_q[kQueue];                 // triangle of the CTA | y - y0 | x - x0 | open coverage
    __shared__ int s_n, s_x0[kRasterThreads], s_y0[kRasterThreads], s_id[3][kRasterThreads];
    __shared__ float s_zlow[kRasterThreads];
    __shared__ double s_plane[kRasterThreads][4];
    const int tid = threadIdx.x;
    const int64_t t = (int64_t)blockIdx.x * kRasterThreads + tid;
    if (tid == 0) s_n = 0;
    __syncthreads();
    bool any = false;
    int id[3] = {0, 0, 0};
    float4 C[3];
    bool draw = t < nt;
    if (draw) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            id[m] = tris[3 * t + m];
            draw = draw && id[m] >= 0 && id[m] < nv;
        }
    }
    bool exact = false;
    if (draw) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            C[m] = xyz[id[m]];
            draw = draw && C[m].w != kVertSkip;
            exact = exact || C[m].w != kVertFast;
        }
    }
    if (draw && exact) {
        raster_exact(cam, verts, tris, t, nv, zkey, big, nbig);
        draw = false;
    }
    if (draw) {
        // positions relative to the whole pixel of vertex 0
        float X[3], Y[3];
        const float4 P0 = at[id[0]], P1 = at[id[1]], P2 = at[id[2]];
        const int ox = __float_as_int(P0.x), oy = __float_as_int(P0.y);
        X[0] = P0.z;
        Y[0] = P0.w;
        X[1] = (float)(__float_as_int(P1.x) - ox) + P1.z;
        Y[1] = (float)(__float_as_int(P1.y) - oy) + P1.w;
        X[2] = (float)(__float_as_int(P2.x) - ox) + P2.z;
        Y[2] = (float)(__float_as_int(P2.y) - oy) + P2.w;
        const float xlo = fminf(fminf(X[0], X[1]), X[2]), xhi = fmaxf(fmaxf(X[0], X[1]), X[2]);
        const float ylo = fminf(fminf(Y[0], Y[1]), Y[2]), yhi = fmaxf(fmaxf(Y[0], Y[1]), Y[2]);
        const float D = fmaxf(fmaxf(xhi, yhi), -fminf(xlo, ylo)) + 1.f;      // > every coordinate used below
        // > the error of X, Y: 6e-8 of the vertex and 2^-24 (D - 1) of the sum
        const float e = 1e-7f * D;
        // pixel centres the box can hold, widened by that error
        const int x0 = max(ox + (int)ceilf(xlo - 2.f * e), 0), x1 = min(ox + (int)floorf(xhi + 2.f * e), cam.w - 1);
        const int y0 = max(oy + (int)ceilf(ylo - 2.f * e), 0), y1 = min(oy + (int)floorf(yhi + 2.f * e), cam.h - 1);
        if (x1 >= x0 && y1 >= y0) {
            if ((int64_t)(x1 - x0 + 1) * (y1 - y0 + 1) > kBigPx) {
                big[atomicAdd(nbig, 1)] = (int)t;
            } else {
                const float X1 = X[1] - X[0], Y1 = Y[1] - Y[0], X2 = X[2] - X[0], Y2 = Y[2] - Y[0];
                // |edge function error| <= tol: its factors are at most 2 D and off
                // by at most 7 e after their differences (44 e D for the two
                // products), and products and difference round (10 e D)
                const float tol = 64.f * e * D;
                // nothing nearer than the nearest vertex is hit, unless the plane
                // is seen edge-on or the triangle is a sliver
                float zlow = -1.f;
                {
                    const float ax = C[1].x - C[0].x, ay = C[1].y - C[0].y, az = C[1].z - C[0].z;
                    const float bx = C[2].x - C[0].x, by = C[2].y - C[0].y, bz = C[2].z - C[0].z;
                    const float nx = ay * bz - az * by, ny = az * bx - ax * bz, nz = ax * by - ay * bx;
                    const float nn = nx * nx + ny * ny + nz * nz;
                    const float l2 = fmaxf(ax * ax + ay * ay + az * az, bx * bx + by * by + bz * bz);
                    float r2 = 0.f;
#pragma unroll
                    for (int m = 0; m < 3; ++m) r2 = fmaxf(r2, C[m].x * C[m].x + C[m].y * C[m].y + C[m].z * C[m].z);
                    const float d = nx * C[0].x + ny * C[0].y + nz * C[0].z;
                    if (nn >= 1e-4f * l2 * l2 && l2 >= 1e-6f * r2 && d * d >= 0.01f * nn * r2)
                        zlow = fminf(fminf(C[0].z, C[1].z), C[2].z) * (1.f - 1e-5f);
                }
                s_zlow[tid] = zlow;
                s_x0[tid] = x0;
                s_y0[tid] = y0;
#pragma unroll
                for (int m = 0; m < 3; ++m) s_id[m][tid] = id[m];
                for (int py = y0; py <= y1; ++py) {
                    const float qy = (float)(py - oy) - Y[0];
                    for (int px = x0; px <= x1; ++px) {
                        const float qx = (float)(px - ox) - X[0];
                        const float f0 = X1 * qy - Y1 * qx;
                        const float f1 = (X2 - X1) * (qy - Y1) - (Y2 - Y1) * (qx - X1);
                        const float f2 = Y2 * (qx - X2) - X2 * (qy - Y2);
                        const float lo = fminf(fminf(f0, f1), f2), hi = fmaxf(fmaxf(f0, f1), f2);
                        if (lo < -tol && hi > tol) continue;
                        if (zlow > 0.f) {
                            const unsigned cur = (unsigned)(__ldcg(zkey + (int64_t)py * cam.w + px) >> 32);
                            if (cur != 0xffffffffu && zlow > __uint_as_float(cur)) continue;
                        }
                        const unsigned open = !(lo > tol || hi < -tol);
                        const int slot = atomicAdd(&s_n, 1);
                        if (slot < kQueue) {
                            s_q[slot] = ((unsigned)tid << 21) | ((unsigned)(py - y0) << 11) | ((unsigned)(px - x0) << 1) | open;
                            any = true;
                        } else if (!open || covered_exact(cam, vd, id[0], id[1], id[2], px, py)) {
                            double n[4];
                            plane_exact(vd, id[0], id[1], id[2], n);
                            depth_exact(cam, n, px, py, slope, (unsigned long long)t, zkey);
                        }
                    }
                }
            }
        }
    }
    if (any) plane_exact(vd, id[0], id[1], id[2], s_plane[tid]);
    __syncthreads();
    const int n = min(s_n, kQueue);
    for (int k = tid; k < n; k += kRasterThreads) {
        const unsigned q = s_q[k];
        const int m = q >> 21;
        const int py = s_y0[m] + (int)((q >> 11) & 1023u), px = s_x0[m] + (int)((q >> 1) & 1023u);
        if (s_zlow[m] > 0.f) {                       // written since?
            const unsigned cur = (unsigned)(__ldcg(zkey + (int64_t)py * cam.w + px) >> 32);
            if (cur != 0xffffffffu && s_zlow[m] > __uint_as_float(cur)) continue;
        }
        if ((q & 1u) && !covered_exact(cam, vd, s_id[0][m], s_id[1][m], s_id[2][m], px, py)) continue;
        depth_exact(cam, s_plane[m], px, py, slope, (unsigned long long)blockIdx.x * kRasterThreads + m, zkey);
    }
}

// The listed large triangles, one CTA each (grid-stride over the list): the
// CTA's threads share the triangle's pixel centres.
__global__ void __launch_bounds__(256) k_raster_big(CamDev cam, const float* __restrict__ verts,
                                                    const int32_t* __restrict__ tris, int64_t nv,
                                                    unsigned long long* __restrict__ zkey,
                                                    const int* __restrict__ big, const int* __restrict__ nbig) {
    const int n = *nbig;
    for (int j = blockIdx.x; j < n; j += gridDim.x) {
        const int64_t t = big[j];
        TriSetup s;
        if (!tri_setup(cam, verts, tris, t, nv, s)) continue;    // always drawn: listed by k_raster
        const int64_t wx = (int64_t)(s.x1 - s.x0) + 1, hy = (int64_t)(s.y1 - s.y0) + 1;
        for (int64_t k = threadIdx.x; k < wx * hy; k += blockDim.x) {
            const double py = s.y0 + (double)(k / wx), px = s.x0 + (double)(k % wx);
            const double dy = dd(ds(py, cam.K[5]), cam.K[4]);
            tri_pixel(cam, s, px, py, dy, (unsigned long long)t, zkey);
        }
    }
}

__device__ __forceinline__ void cam_point_f(const CamDev& c, const float* X, float xc[3]) {
#pragma unroll
    for (int r = 0; r < 3; ++r)
        xc[r] = c.RTf[4 * r] * X[0] + c.RTf[4 * r + 1] * X[1] + c.RTf[4 * r + 2] * X[2] + c.RTf[4 * r + 3];
}

__device__ __forceinline__ float dot_cross(const float n[3], const float a[3], const float b[3]) {
    // n . (a x b)
    return n[0] * (a[1] * b[2] - a[2] * b[1]) + n[1] * (a[2] * b[0] - a[0] * b[2]) +
           n[2] * (a[0] * b[1] - a[1] * b[0]);
}

__device__ __forceinline__ void bilinear(const uint8_t* img, int w, int h, float u, float v, float out[3]) {
    const float fu = floorf(u), fv = floorf(v);
    const int x0 = (int)fu, y0 = (int)fv;
    const float fx = u - fu, fy = v - fv;
    const int xa = min(max(x0, 0), w - 1), xb = min(max(x0 + 1, 0), w - 1);
    const int ya = min(max(y0, 0), h - 1), yb = min(max(y0 + 1, 0), h - 1);
    const uint8_t* p00 = img + 3 * ((int64_t)ya * w + xa);
    const uint8_t* p10 = img + 3 * ((int64_t)ya * w + xb);
    const uint8_t* p01 = img + 3 * ((int64_t)yb * w + xa);
    const uint8_t* p11 = img + 3 * ((int64_t)yb * w + xb);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        out[c] = (1.f - fx) * (1.f - fy) * p00[c] + fx * (1.f - fy) * p10[c] + (1.f - fx) * fy * p01[c] +
                 fx * fy * p11[c];
}

__global__ void __launch_bounds__(256) k_resolve(CamDev cam, const float* __restrict__ verts,
                                                 const int32_t* __restrict__ tris,
                                                 const unsigned long long* __restrict__ zkey,
                                                 float* __restrict__ depth, uint8_t* __restrict__ rgb,
                                                 const uint8_t* __restrict__ vrgb, const float* __restrict__ tw,
                                                 const float* __restrict__ tuv, TexDev tex) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t npx = (int64_t)cam.w * cam.h;
    if (p >= npx) return;
    const unsigned long long key = zkey[p];
    if (key == ~0ull) {
        depth[p] = 0.f;
        if (rgb) rgb[3 * p] = rgb[3 * p + 1] = rgb[3 * p + 2] = 0;
        return;
    }
    const float z = __uint_as_float((unsigned)(key >> 32));
    depth[p] = z;
    if (!rgb) return;
    const int64_t t = (int64_t)(key & 0xffffffffull);
    const int ia = tris[3 * t], ib = tris[3 * t + 1], ic = tris[3 * t + 2];
    float A[3], B[3], C[3];
    cam_point_f(cam, verts + 3 * (int64_t)ia, A);
    cam_point_f(cam, verts + 3 * (int64_t)ib, B);
    cam_point_f(cam, verts + 3 * (int64_t)ic, C);
    const float py = (float)(p / cam.w), px = (float)(p % cam.w);
    const float dy = (py - cam.Kf[5]) / cam.Kf[4];
    const float dx = ((px - cam.Kf[2]) - cam.Kf[1] * dy) / cam.Kf[0];
    const float P[3] = {z * dx, z * dy, z};
    float e1[3], e2[3], n[3], pa[3], pb[3], pc[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        e1[r] = B[r] - A[r];
        e2[r] = C[r] - A[r];
        pa[r] = A[r] - P[r];
        pb[r] = B[r] - P[r];
        pc[r] = C[r] - P[r];
    }
    n[0] = e1[1] * e2[2] - e1[2] * e2[1];
    n[1] = e1[2] * e2[0] - e1[0] * e2[2];
    n[2] = e1[0] * e2[1] - e1[1] * e2[0];
    const float nn = n[0] * n[0] + n[1] * n[1] + n[2] * n[2];
    const float la = dot_cross(n, pb, pc) / nn;
    const float lb = dot_cross(n, pc, pa) / nn;
    const float lc = dot_cross(n, pa, pb) / nn;
    float col[3] = {0.f, 0.f, 0.f};
    if (vrgb) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            col[c] = la * vrgb[3 * ia + c] + lb * vrgb[3 * ib + c] + lc * vrgb[3 * ic + c];
    } else if (tw) {
        const int K = tex.k;
        float acc[3] = {0.f, 0.f, 0.f}, wsum = 0.f;
        for (int k = 0; k < K; ++k) {
            const float wa = tw[(int64_t)ia * K + k], wb = tw[(int64_t)ib * K + k], wc = tw[(int64_t)ic * K + k];
            if (!(wa > 0.f && wb > 0.f && wc > 0.f)) continue;
            const float wk = la * wa + lb * wb + lc * wc;
            const float uk = la * tuv[2 * ((int64_t)ia * K + k)] + lb * tuv[2 * ((int64_t)ib * K + k)] +
                             lc * tuv[2 * ((int64_t)ic * K + k)];
            const float vk = la * tuv[2 * ((int64_t)ia * K + k) + 1] + lb * tuv[2 * ((int64_t)ib * K + k) + 1] +
                             lc * tuv[2 * ((int64_t)ic * K + k) + 1];
            float s[3];
            bilinear(tex.rgb[k], tex.rgb_w[k], tex.rgb_h[k], uk, vk, s);
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[c] += wk * s[c];
            wsum += wk;
        }
        if (wsum > 0.f) {
#pragma unroll
            for (int c = 0; c < 3; ++c) col[c] = acc[c] / wsum;
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) rgb[3 * p + c] = (uint8_t)fminf(fmaxf(floorf(col[c] + 0.5f), 0.f), 255.f);
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

CamDev make_cam(const ftr_camera& c) {
    CamDev d{};
    d.w = c.w;
    d.h = c.h;
    for (int j = 0; j < 9; ++j) d.K[j] = d.Kf[j] = c.K[j];
    for (int j = 0; j < 12; ++j) d.RT[j] = d.RTf[j] = c.world_to_cam[j];
    return d;
}

}  // namespace

bool camera_ok(const ftr_camera* cam) {
    return cam && cam->w >= 1 && cam->h >= 1 && cam->w <= 16384 && cam->h <= 16384 && cam->K[0] != 0.f &&
           cam->K[4] != 0.f;
}

}  // namespace ftr

using namespace ftr;

int ftr_render(ftr_ctx* c, const ftr_render_src* src, const ftr_camera* cam, float* depth_out, uint8_t* rgb_out) {
    if (!c) return FTR_EINVAL;
    if (!src || !camera_ok(cam) || !depth_out)
        return set_err(c, FTR_EINVAL, "ftr_render: a source, a camera (w, h in 1..16384, focal != 0) and depth_out");
    if (src->n_tris < 0 || src->n_tris >= (int64_t)1 << 31 || src->n_vertices < 0)
        return set_err(c, FTR_EINVAL, "ftr_render: 0 <= n_tris < 2^31");
    if (src->vertex_rgb && src->tex_weights)
        return set_err(c, FTR_EINVAL, "ftr_render: one colour source at most");
    if ((src->vertex_rgb || src->tex_weights) && !rgb_out)
        return set_err(c, FTR_EINVAL, "ftr_render: a colour source needs rgb_out");
    if (!dev_ptr(depth_out) || (rgb_out && !dev_ptr(rgb_out)))
        return set_err(c, FTR_EINVAL, "ftr_render: outputs must be device memory");
    if (src->n_tris > 0 && (!dev_ptr(src->vertices) || !dev_ptr(src->tris)))
        return set_err(c, FTR_EINVAL, "ftr_render: vertices and tris must be device memory");
    if (src->vertex_rgb && !dev_ptr(src->vertex_rgb))
        return set_err(c, FTR_EINVAL, "ftr_render: vertex_rgb must be device memory");
    TexDev tex{};
    if (src->tex_weights) {
        if (src->tex_k < 1 || src->tex_k > kMaxViews || !src->tex_views || !dev_ptr(src->tex_weights) ||
            !dev_ptr(src->tex_uv))
            return set_err(c, FTR_EINVAL, "ftr_render: 1 <= tex_k <= 8 views, device weights and uv");
        tex.k = src->tex_k;
        for (int k = 0; k < tex.k; ++k) {
            const ftr_view& v = src->tex_views[k];
            if (v.rgb_w < 1 || v.rgb_h < 1 || !dev_ptr(v.rgb))
                return set_err(c, FTR_EINVAL, "ftr_render: view %d needs a device RGB image", k);
            tex.rgb_w[k] = v.rgb_w;
            tex.rgb_h[k] = v.rgb_h;
            tex.rgb[k] = v.rgb;
        }
    }
    EvalScratch* ev = eval_scratch(c);
    if (!ev) return set_err(c, FTR_ENOMEM, "ftr_render: scratch");
    const int64_t npx = (int64_t)cam->w * cam->h;
    cudaError_t e;
    if (npx > ev->zkey_cap) {
        cudaStreamSynchronize(c->stream);
        if (ev->zkey) cudaFree(ev->zkey);
        ev->zkey = nullptr;
        ev->zkey_cap = 0;
        if ((e = cudaMalloc((void**)&ev->zkey, (size_t)npx * sizeof(unsigned long long))) != cudaSuccess)
            return cuda_fail(c, e, "ftr_render: z-buffer");
        ev->zkey_cap = npx;
    }
    if (src->n_tris + 1 > ev->big_cap) {
        cudaStreamSynchronize(c->stream);
        if (ev->big) cudaFree(ev->big);
        ev->big = nullptr;
        ev->big_cap = 0;
        if ((e = cudaMalloc((void**)&ev->big, (size_t)(src->n_tris + 1) * sizeof(int))) != cudaSuccess)
            return cuda_fail(c, e, "ftr_render: triangle list");
        ev->big_cap = src->n_tris + 1;
    }
    const CamDev cd = make_cam(*cam);
    if ((e = cudaMemsetAsync(ev->zkey, 0xff, (size_t)npx * sizeof(unsigned long long), c->stream)) != cudaSuccess)
        return cuda_fail(c, e, "ftr_render: clear");
    if (src->n_tris > 0) {
        int* nbig = ev->big + src->n_tris;
        if ((e = cudaMemsetAsync(nbig, 0, sizeof(int), c->stream)) != cudaSuccess)
            return cuda_fail(c, e, "ftr_render: clear");
        // scratch: at, xyz, vd (3 doubles per vertex), slopes (w + h doubles).
        // n_vertices may be no more than a bound: k_project reads every vertex up to
        // it, so it runs only where they all lie in the array's allocation and where
        // triangles that share no vertex would name as many; else each triangle reads
        // its own three.
        const int64_t nv = src->n_vertices, nslope = (int64_t)cam->w + cam->h;
        const size_t need = (size_t)nv * (16 + 16 + 24) + (size_t)nslope * 8;
        bool project = nv <= 3 * src->n_tris && room_behind(src->vertices) >= (size_t)nv * 3 * sizeof(float);
        if (project && need > ev->proj_cap) {
            cudaStreamSynchronize(c->stream);
            if (ev->proj) cudaFree(ev->proj);
            ev->proj = nullptr;
            ev->proj_cap = 0;
            if (cudaMalloc(&ev->proj, need) == cudaSuccess) {
                ev->proj_cap = need;
            } else {
                cudaGetLastError();
                ev->proj = nullptr;
                project = false;
            }
        }
        const unsigned blocks = (unsigned)((src->n_tris + kRasterThreads - 1) / kRasterThreads);
        if (project) {
            float4* at = static_cast<float4*>(ev->proj);
            float4* xyz = at + nv;
            double* vd = reinterpret_cast<double*>(xyz + nv);
            double* slope = vd + 3 * nv;
            k_project<<<(unsigned)((nv + nslope + 255) / 256), 256, 0, c->stream>>>(cd, src->vertices, nv, at, xyz,
                                                                                    vd, slope);
            c->launches++;
            k_raster<<<blocks, kRasterThreads, 0, c->stream>>>(cd, src->vertices, src->tris, src->n_tris, nv, at, xyz,
                                                               vd, slope, ev->zkey, ev->big, nbig);
        } else {
            k_raster_exact<<<blocks, kRasterThreads, 0, c->stream>>>(cd, src->vertices, src->tris, src->n_tris, nv,
                                                                     ev->zkey, ev->big, nbig);
        }
        k_raster_big<<<2 * kSms, 256, 0, c->stream>>>(cd, src->vertices, src->tris, src->n_vertices, ev->zkey, ev->big,
                                                     nbig);
        c->launches += 2;
        if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(c, e, "ftr_render: raster");
    }
    k_resolve<<<(unsigned)((npx + 255) / 256), 256, 0, c->stream>>>(
        cd, src->vertices, src->tris, ev->zkey, depth_out, rgb_out, src->vertex_rgb, src->tex_weights,
        src->tex_uv, tex);
    c->launches++;
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(c, e, "ftr_render: resolve");
    return FTR_OK;
}

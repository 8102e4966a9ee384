// Splat of oriented points into the gradient field V (Sec. III-B, eq. 1-2).
//
//   U(q) = sum_i g(|X_i - p(q)|; sigma1) W_i N_i,  d(q) = sum_i g(|X_i - p(q)|; sigma2) W_i
//   g(x; s) = s^-1 exp(-x^2 / s^2),                V(q) = U(q) / d(q)
//
// over the 4^3 nodes floor(t)-1 .. floor(t)+2 around each point.  The grid is
// cut into 8^3-node bricks; only bricks touched by some stencil get storage.
// Per frame:
//   ingest  point -> (floor t, t - floor t, W, N); t as a float pair, the
//           float64 path only within 1e-5 of a decision; an accepted point
//           adds 1 to every brick its stencil overlaps (counts zeroed when
//           the frame is reset)
//   scan    256-brick tiles: per-tile sums, then each tile adds the sums
//           before it and writes brick offsets, a dense slot per touched
//           brick and the accumulation chunks (no single-CTA scan)
//   fill    per point, append its index to each overlapped brick's list
//   accum   persistent CTAs take work units (up to 1024 (point, brick) pairs
//           of one touched brick): a warp per pair evaluates the stencil nodes
//           inside the brick and adds the contributions to shared-memory
//           fixed-point accumulators (value * 2^40 as 32-bit hi/lo halves, exact
//           and order-independent, so the result is bit-reproducible; 64-bit in
//           a frame with weights or normals beyond their range); a brick of several units adds each
//           unit's exact sums into an int64 global accumulator and its last
//           unit writes V = (sigma2 / sigma1) U / d to the brick's slot.
// The simple variant (nearest node floor(t + 1/2), V = mean N) uses the same
// bricks with one node per point and d counting points.
#include <cuda_runtime.h>
#include <math.h>

#include "ftr_internal.h"
#include "node_pos.cuh"

namespace ftr {

namespace {

// Brick range [lo, hi] per axis that the point's stencil overlaps.
__device__ __forceinline__ bool stencil_bricks(const int4 b, int mode, int lo[3], int hi[3]) {
    if (!(b.w & 1)) return false;
    const int bb[3] = {b.x, b.y, b.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (mode == FTR_SPLAT_WEIGHTED) {
            lo[c] = (bb[c] - 1) >> 3;
            hi[c] = (bb[c] + 2) >> 3;
        } else {
            int node = bb[c] + ((b.w >> (1 + c)) & 1);
            lo[c] = hi[c] = node >> 3;
        }
    }
    return true;
}

// Runs of equal b over the lanes of a full warp: the first lane of this lane's
// run and the run's length.  Consecutive points are neighbouring pixels, mostly
// in the same bricks, so one atomic per run serves almost as few addresses as
// one per distinct value, for a shuffle and a ballot (a match over the warp
// takes a step per distinct value: 8 of them were half of this stage).
struct Run {
    int first, len;
};
__device__ __forceinline__ Run run_of(int b, int lane) {
    const int prev = __shfl_up_sync(0xffffffffu, b, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || prev != b);
    const unsigned upto = heads & (0xffffffffu >> (31 - lane)), after = heads & ~(0xffffffffu >> (31 - lane));
    Run r;
    r.first = 31 - __clz(upto);
    r.len = (after ? __ffs(after) - 1 : 32) - r.first;
    return r;
}

constexpr float kTameNormal = 1.99f;   // normal components below it: 1024 x (1.99 2^20 + 1/2) < 2^31
static_assert(kSplatChunk <= 1024, "the sums of one unit fit the 32-bit halves");

// One point: t per axis with every decision equal to the float64 one, the
// acceptance test, and the point record at slot `dst`.
// An accepted point also counts itself into every brick its stencil overlaps
// (cnt: per-brick point counts of the frame, zeroed when the frame starts).
// Called by whole warps; lanes without a point have live = false.
__device__ __forceinline__ void ingest_one(bool live, const float* p, const float* q, const float* wp, int64_t dst, const GridDev& g,
                                           int4* pbase, float4* pfrac, float4* pnrm, unsigned long long* dropped,
                                           int* wild, int* cnt) {
    bool ok = live;
    int fl[3] = {0, 0, 0};
    float fr[3] = {0.f, 0.f, 0.f};
    float x3[3] = {0.f, 0.f, 0.f}, q3[3] = {0.f, 0.f, 0.f}, wi = 1.f;
    if (live) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x3[c] = p[c];
            q3[c] = q[c];
        }
        if (wp) wi = *wp;
    }
    int up = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (!live) break;
        const float x = x3[c];
        int fli;
        float r;
        bool u;
        if (node_t_pair(x, g.bminf[c], g.inv_hf[c], g.inv_h_lo[c], fli, r, u)) {
            const bool in = fli >= 1 && fli <= g.n[c] - 3;   // 1 <= t < n - 2
            ok = ok && in;
            if (in) {
                fl[c] = fli;
                fr[c] = r;
                if (u) up |= 1 << c;
            }
        } else {
            const double t = node_t((double)x, g.bmin[c], g.h[c], g.inv_h[c], (double)g.n[c]);
            const bool in = (t >= 1.0) && (t < (double)g.n[c] - 2.0);   // false for NaN
            ok = ok && in;
            if (in) {
                const double f = floor(t);
                fl[c] = (int)f;
                fr[c] = (float)(t - f);
                if (floor(t + 0.5) > f) up |= 1 << c;
            }
        }
    }
    if (!ok) {
        if (live) atomicAdd(dropped, 1ull);
        fl[0] = fl[1] = fl[2] = 0;
    }
    const int4 rec = make_int4(fl[0], fl[1], fl[2], ok ? (1 | (up << 1)) : 0);
    // per brick slot k of the at most 2 x 2 x 2 bricks the stencil overlaps, a
    // run of lanes counting into the same brick adds its length with one atomic
    const int lane = threadIdx.x & 31;
    const int shift = count_shift(g.nb[0] * g.nb[1] * g.nb[2]);
    int lo[3] = {0, 0, 0}, hi[3] = {-1, -1, -1};
    const bool any = stencil_bricks(rec, g.mode, lo, hi);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int bx = lo[0] + (k & 1), by = lo[1] + ((k >> 1) & 1), bz = lo[2] + (k >> 2);
        const bool valid = any && bx <= hi[0] && by <= hi[1] && bz <= hi[2];
        const int b = valid ? bx + g.nb[0] * (by + g.nb[1] * bz) : -1;
        const Run r = run_of(b, lane);
        if (valid && lane == r.first) atomicAdd(&cnt[b << shift], r.len);
    }
    if (!live) return;
    pbase[dst] = rec;
    // outside the range of the accumulation's 32-bit halves: kSplatChunk contributions
    // of a component below 2 can all fall on one node
    const bool tame = wi >= 0.f && wi <= 1.f && fabsf(q3[0]) < kTameNormal && fabsf(q3[1]) < kTameNormal &&
                      fabsf(q3[2]) < kTameNormal;
    if (ok && !tame) atomicOr(wild, 1);
    pfrac[dst] = make_float4(fr[0], fr[1], fr[2], wi);
    pnrm[dst] = make_float4(q3[0], q3[1], q3[2], 0.f);
}

// n_dev (nullable): the point count on the device; n then only bounds it.
__global__ void k_ingest(const float* __restrict__ pts, const float* __restrict__ nrm,
                         const float* __restrict__ w, int64_t n, int64_t base, GridDev g, int4* pbase,
                         float4* pfrac, float4* pnrm, unsigned long long* dropped, int* wild,
                         int64_t* npts_dev, const int* __restrict__ n_dev, int* cnt) {
    pdl_wait();
    if (n_dev) n = min(n, (int64_t)*n_dev);
    if (blockIdx.x == 0 && threadIdx.x == 0) *npts_dev = base + n;   // points stored so far: later kernels read it here
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < n; i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + threadIdx.x;
        ingest_one(i < n, pts + 3 * i, nrm + 3 * i, w ? w + i : nullptr, base + i, g, pbase, pfrac, pnrm, dropped,
                   wild, cnt);
    }
}

// Several point sets in one launch: thread i ingests point i of the
// concatenation of the sets (set order, as separate launches would store them).
__global__ void k_ingest_sets(IngestSets S, GridDev g, int4* pbase, float4* pfrac, float4* pnrm,
                              unsigned long long* dropped, int* wild, int64_t* npts_dev, int* cnt) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *npts_dev = S.base + S.off[S.k];
    int s = 0;
    while (s + 1 < S.k && i >= S.off[s + 1]) ++s;
    const int64_t j = i - S.off[s];
    ingest_one(i < S.off[S.k], S.pts[s] + 3 * j, S.nrm[s] + 3 * j, S.w[s] ? S.w[s] + j : nullptr, S.base + i, g, pbase, pfrac, pnrm,
               dropped, wild, cnt);
}

// Grid-stride over the stored points; the count is read on the device, so the
// launch does not depend on it.
// A warp takes 32 consecutive points (neighbouring pixels of one camera,
// mostly the same bricks): per brick slot k of the at most 2 x 2 x 2 bricks
// a stencil overlaps, a run of lanes that append to the same brick reserves its
// places with one atomic (the first lane's) and each writes at its rank.  The
// atomics of the eight slots are all issued before the first place is used:
// one after another, their round trips made this pass 7-12 us.
__global__ void k_brick_fill(const int4* __restrict__ pbase, const int64_t* __restrict__ npts, GridDev g,
                             int* cursor, int* entries) {
    pdl_wait();
    const int64_t n = *npts;
    const int lane = threadIdx.x & 31;
    const int shift = count_shift(g.nb[0] * g.nb[1] * g.nb[2]);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform loop: every lane reaches each match below
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n; i0 += stride) {
        const int64_t i = i0 + lane;
        int lo[3] = {0, 0, 0}, hi[3] = {-1, -1, -1};
        const bool ok = i < n && stencil_bricks(pbase[i], g.mode, lo, hi);
        Run run[8];
        int pos[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int bx = lo[0] + (k & 1), by = lo[1] + ((k >> 1) & 1), bz = lo[2] + (k >> 2);
            const bool valid = ok && bx <= hi[0] && by <= hi[1] && bz <= hi[2];
            const int b = valid ? bx + g.nb[0] * (by + g.nb[1] * bz) : -1;
            run[k] = run_of(b, lane);
            pos[k] = 0;
            if (valid && lane == run[k].first) pos[k] = atomicAdd(&cursor[b << shift], run[k].len);
            if (!valid) run[k].len = 0;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int at = __shfl_sync(0xffffffffu, pos[k], run[k].first);
            if (run[k].len) entries[at + lane - run[k].first] = (int)i;
        }
    }
}

// Exclusive scan of the brick counts in three coalesced launches over tiles
// of kTile bricks: (1) per-tile sums of the counts and of the touched
// bricks, (2) each tile adds up the sums before it, rescans itself with
// that offset and writes the fill cursors, the dense slot of every touched
// brick (-1 otherwise), the accumulation units and the z-range.
constexpr int kScanT = 256;
constexpr int kTile = kBrickScanTile;
static_assert(kTile % kScanT == 0, "a tile is a whole number of block scans");
// A brick's pairs are accumulated in chunks of at most kChunk (point, brick)
// pairs, one chunk per CTA at a time; the 32-bit hi/lo accumulators hold that many
// contributions of weight 1 and a normal component below 1.99 on one voxel.
constexpr int kChunk = kSplatChunk;
constexpr int kHeavyUnit = 1 << 30;   // the unit's brick has more than one chunk

// Block-wide exclusive scan of four ints per thread (kScanT threads).
__device__ __forceinline__ int4 block_scan4(int4 v, int4& total, int4* sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int4 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, inc.x, o);
        const int b = __shfl_up_sync(0xffffffffu, inc.y, o);
        const int c = __shfl_up_sync(0xffffffffu, inc.z, o);
        const int d = __shfl_up_sync(0xffffffffu, inc.w, o);
        if (lane >= o) {
            inc.x += a;
            inc.y += b;
            inc.z += c;
            inc.w += d;
        }
    }
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int4 w = lane < kScanT / 32 ? sh[lane] : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, w.x, o);
            const int b = __shfl_up_sync(0xffffffffu, w.y, o);
            const int c = __shfl_up_sync(0xffffffffu, w.z, o);
            const int d = __shfl_up_sync(0xffffffffu, w.w, o);
            if (lane >= o) {
                w.x += a;
                w.y += b;
                w.z += c;
                w.w += d;
            }
        }
        if (lane < kScanT / 32) sh[lane] = w;
    }
    __syncthreads();
    const int4 before = wid ? sh[wid - 1] : make_int4(0, 0, 0, 0);
    total = sh[kScanT / 32 - 1];
    __syncthreads();
    return make_int4(before.x + inc.x - v.x, before.y + inc.y - v.y, before.z + inc.z - v.z,
                     before.w + inc.w - v.w);
}

// Per brick of c (point, brick) pairs: (pairs, touched, accumulation chunks,
// heavy = more than one chunk).
__device__ __forceinline__ int4 brick_counts(int c) {
    const int ch = (c + kChunk - 1) / kChunk;
    return make_int4(c, c > 0, ch, ch > 1);
}

// Size class of a unit of n pairs: 32 pairs wide (the last: 993 to kChunk).
__device__ __forceinline__ int size_class(int n) { return min((n - 1) >> 5, kSizeClasses - 1); }

__global__ void __launch_bounds__(kScanT) k_brick_tile_sums(const int* __restrict__ cnt, int nb, int4* tile_sum,
                                                            int* meta) {
    pdl_wait();
    __shared__ int4 sh[kScanT / 32];
    __shared__ int s_class[kSizeClasses];
    if (threadIdx.x < kSizeClasses) s_class[threadIdx.x] = 0;
    __syncthreads();
    int4 v = make_int4(0, 0, 0, 0);
    for (int k = 0; k < kTile / kScanT; ++k) {
        const int b = blockIdx.x * kTile + k * kScanT + threadIdx.x;
        if (b < nb) {
            const int4 q = brick_counts(cnt[b << count_shift(nb)]);
            v.x += q.x;
            v.y += q.y;
            v.z += q.z;
            v.w += q.w;
            if (q.z > 1) atomicAdd(&s_class[kSizeClasses - 1], q.z - 1);   // full chunks
            if (q.z > 0) atomicAdd(&s_class[size_class(q.x - (q.z - 1) * kChunk)], 1);
        }
    }
    int4 tot;
    block_scan4(v, tot, sh);
    if (threadIdx.x < kSizeClasses && s_class[threadIdx.x])
        atomicAdd(&meta[kMetaClasses + threadIdx.x], s_class[threadIdx.x]);
    if (threadIdx.x == 0) {
        tile_sum[blockIdx.x] = tot;
        if (blockIdx.x == 0) {       // the z range is min/max-reduced by the write kernel
            meta[2] = 0x7fffffff;
            meta[3] = -1;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < kMetaClasses - kMetaRows) meta[kMetaRows + threadIdx.x] = 0;   // live rows: or-ed
}

// Per tile: its exclusive offset is the sum of the (few) tile sums before it,
// summed by every CTA itself (no separate scan launch); CTA 0 also writes the
// totals.  Then the tile's bricks get their offsets, slots and chunk ranges.
__global__ void __launch_bounds__(kScanT) k_brick_tile_write(const int* __restrict__ cnt, int nb, int nbx, int nbxy,
                                                             const int4* __restrict__ tile_sum, int ntiles,
                                                             int* cursor, int* slot, int* meta,
                                                             int* unit_off, int* heavy_idx, int4* units) {
    pdl_wait();
    __shared__ int4 sh[kScanT / 32];
    // units of this tile per size class, then where they go: after the larger
    // classes' units and the units of its class that other tiles placed first
    __shared__ int s_class[kSizeClasses];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < kSizeClasses) s_class[threadIdx.x] = 0;
    int4 pre = make_int4(0, 0, 0, 0), all = make_int4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < ntiles; i += kScanT) {
        const int4 v = tile_sum[i];
        if (i < (int)blockIdx.x) {
            pre.x += v.x;
            pre.y += v.y;
            pre.z += v.z;
            pre.w += v.w;
        }
        all.x += v.x;
        all.y += v.y;
        all.z += v.z;
        all.w += v.w;
    }
    int4 run, total;
    block_scan4(pre, run, sh);
    block_scan4(all, total, sh);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        unit_off[total.y] = total.z;   // end of the last touched brick's chunks
        meta[0] = total.y;
        meta[1] = total.x;
        meta[4] = 0;                   // chunk ticket of the accumulation
        meta[5] = total.z;             // chunks in all
        meta[6] = total.w;             // heavy bricks
    }
    static_assert(kTile == kScanT, "a thread per brick");
    int zmin = 0x7fffffff, zmax = -1;
    const int shift = count_shift(nb);
    {
        const int b = blockIdx.x * kTile + threadIdx.x;
        const int c = b < nb ? cnt[b << shift] : 0;
        const int4 q = brick_counts(c);
        // rank of the brick's full chunks and of its last chunk in their classes
        const int nlast = c - (q.z - 1) * kChunk;
        int rfull = 0, rlast = 0;
        if (q.z > 1) rfull = atomicAdd(&s_class[kSizeClasses - 1], q.z - 1);
        if (q.z > 0) rlast = atomicAdd(&s_class[size_class(nlast)], 1);
        int4 tot;
        const int4 ex = block_scan4(q, tot, sh);
        if (threadIdx.x < kSizeClasses) {
            const int mine = s_class[lane], count = meta[kMetaClasses + lane];
            const int at = mine ? atomicAdd(&meta[kMetaClasses + kSizeClasses + lane], mine) : 0;
            int larger = count;                      // inclusive sum over the classes from this one up
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_down_sync(0xffffffffu, larger, o);
                if (lane + o < 32) larger += v;
            }
            s_class[lane] = larger - count + at;
        }
        __syncthreads();
        if (b < nb) {
            cursor[b << shift] = run.x + ex.x;
            if (c > 0) {
                const int s = run.y + ex.y;
                slot[b] = s;
                unit_off[s] = run.z + ex.z;
                // per chunk all that its CTA needs: brick, slot, first pair, pairs (| kHeavyUnit)
                const int hv = q.w ? kHeavyUnit : 0;
                for (int j = 0; j + 1 < q.z; ++j)
                    units[s_class[kSizeClasses - 1] + rfull + j] = make_int4(b, s, run.x + ex.x + j * kChunk, kChunk | hv);
                units[s_class[size_class(nlast)] + rlast] = make_int4(b, s, run.x + ex.x + (q.z - 1) * kChunk, nlast | hv);
                heavy_idx[s] = q.w ? run.w + ex.w : -1;
                const int bz = b / nbxy;
                zmin = zmax = bz;
                // its pair of brick rows = 16 grid rows; the first brick of a run along x sets the bit
                const int by = (b - bz * nbxy) / nbx;
                if (b % nbx == 0 || cnt[(b - 1) << shift] == 0) atomicOr(&meta[kMetaRows + bz], 1 << (by >> 1));
            } else {
                slot[b] = -1;
            }
        }
    }
    if (zmax >= 0) {
        atomicMin(&meta[2], zmin);
        atomicMax(&meta[3], zmax);
    }
}

constexpr int kAccThreads = 256;

// round(v * 2^40) as int64 without a 64-bit conversion (those run on the slow
// double-precision pipe): with x = v 2^9, hi = trunc(x) and r = x - hi (exact:
// Sterbenz, or r = x when |x| < 1), v 2^40 = hi 2^31 + r 2^31 where r 2^31 is
// an exact float in (-2^31, 2^31) rounded to the nearest integer (ties to
// even, like the direct conversion, since hi 2^31 is even).
__device__ __forceinline__ long long fix40(float v) {
    const float x = v * 512.0f;
    const float hf = truncf(x);
    const int lo = __float2int_rn((x - hf) * 2147483648.0f);
    return (long long)(int)hf * 2147483648ll + (long long)lo;
}

// int64 -> float32 of its magnitude's two 32-bit halves, sign restored after
// (no cancellation for small negative values; no 64-bit conversion)
__device__ __forceinline__ float fix_to_float(long long v) {
    const bool neg = v < 0;
    const unsigned long long m = neg ? (unsigned long long)(-v) : (unsigned long long)v;
    const float f = fmaf((float)(unsigned)(m >> 32), 4294967296.0f, (float)(unsigned)(m & 0xffffffffull));
    return neg ? -f : f;
}

constexpr int kStage = kAccThreads;   // point records staged in shared memory per batch (one per thread)

// Fixed-point contribution round(v * 2^40) = hi 2^20 + lo of |v| < 4: hi = round(v
// 2^20); r = v - hi 2^-20 is exact (Sterbenz, or r = v when hi = 0) with |r| <= 2^-21,
// and lo = round(r 2^40) in [-2^19, 2^19].  Ties go to even as in a direct conversion
// (hi 2^20 is even).  Adding 1.5 2^23 rounds to an integer and leaves it in the low
// mantissa bits: conversions run on a unit with a quarter of the rate.
__device__ __forceinline__ void fix40_split(float v, int& hi, int& lo) {
    constexpr float kMagic = 12582912.0f;
    const float f = __fmaf_rn(v, 1048576.0f, kMagic);
    hi = __float_as_int(f) - __float_as_int(kMagic);
    const float r = __fmaf_rn(__fsub_rn(f, kMagic), -9.5367431640625e-07f, v);
    lo = __float_as_int(__fmaf_rn(r, 1099511627776.0f, kMagic)) - __float_as_int(kMagic);
}

// Accumulator index of brick node li = x + 8 y + 64 z: planes 68 apart, so that
// the 4 x 4 nodes of two adjacent planes that a warp adds to fall on 32
// different banks.
constexpr int kPlane = 68;
constexpr int kAccVox = 8 * kPlane;
__device__ __forceinline__ int acc_of(int li) { return (li & 63) + kPlane * (li >> 6); }

// Persistent CTAs take work units: a unit is one chunk of at most kChunk
// (point, brick) pairs of one touched brick, described by one record.  A warp
// takes a pair: 4 x 4 nodes of two stencil planes per step, over the planes
// that fall inside the brick (2.9 of 4 on average), and adds the fixed-point
// contributions to shared-memory accumulators.  Integer
// sums are exact and order-independent, so V is bit-reproducible.  32-bit
// atomics on the (hi, lo) parts: a chunk has at most kChunk = 1024 points, so with
// weights in [0, 1] and normal components below 1.99 |sum hi| < 2^31 and |sum lo| <=
// 2^29; a frame with a weight or a normal outside takes 64-bit shared atomics
// throughout.  A brick of one chunk writes V directly; the chunks
// of a heavier brick add their exact sums into its int64 accumulator in
// global memory, and the chunk that completes last (a per-brick counter)
// writes V and clears the accumulator for the next frame.
//
// Bricks differ in size by a factor of a hundred, and an SM holds only about
// seven of a 256^3 frame's: in grid order one SM ran 2.4 times the mean.  The
// binning therefore lists the units by size, largest first: unit u < gridDim.x
// belongs to CTA u, so that each SM starts with one of every size, and the
// ticket (zeroed by the binning) gives out the small rest, drawn while the
// current unit runs (256^3 frame: 43 us, now 34).  (Without atomics, each warp owning two planes of the
// brick, the work was less evenly spread within a CTA and took longer.)
template <bool WEIGHTED>
__global__ void __launch_bounds__(kAccThreads, 6) k_splat_accum(GridDev g, int* __restrict__ meta,
                                                                const int4* __restrict__ units,
                                                                const int* __restrict__ entries,
                                                                const int4* __restrict__ pbase,
                                                                const float4* __restrict__ pfrac,
                                                                const float4* __restrict__ pnrm,
                                                                const int* __restrict__ wild,
                                                                float* __restrict__ vpool,
                                                                const int* __restrict__ unit_off,
                                                                const int* __restrict__ heavy_idx,
                                                                unsigned long long* __restrict__ heavy_acc,
                                                                int* __restrict__ heavy_done) {
    pdl_wait();
    __shared__ __align__(16) unsigned acc[8][kAccVox];   // fast: [c] hi, [4 + c] lo; slow: 4 x int64
    __shared__ float4 s_frac[kStage];    // frac + 1 per axis (weighted), W
    __shared__ float4 s_nrm[kStage];     // N, stencil corner in the brick as packed bytes
    __shared__ int s_next;
    __shared__ bool s_last;
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int ox = lane & 3, oy = (lane >> 2) & 3;
    unsigned long long* acc64 = reinterpret_cast<unsigned long long*>(&acc[0][0]);
    const float fox = (float)ox, foy = (float)oy;
    // packed node coordinates: fields at bits 0, 12 and 24, biased by 8, so that
    // a coordinate lies in the brick iff bit 3 is set and bit 4 clear
    const unsigned lane_off = (unsigned)(ox | (oy << 12));
    const bool fast = wild[0] == 0;                                     // block-uniform
    const int nunits = meta[5];
    if (blockIdx.x == 0 && tid < 2 * kSizeClasses) meta[kMetaClasses + tid] = 0;   // for the next frame's binning
    for (int unit = blockIdx.x; unit < nunits;) {
        if (tid == 0) s_next = (int)gridDim.x + atomicAdd(meta + 4, 1);   // needed after this unit
        const int4 U = units[unit];
        const int b = U.x, s = U.y, e0 = U.z, e1 = U.z + (U.w & (kHeavyUnit - 1));
        const bool heavy = (U.w & kHeavyUnit) != 0;
        const int bx = b % g.nb[0], by = (b / g.nb[0]) % g.nb[1], bz = b / (g.nb[0] * g.nb[1]);
        const int orgx = bx * kBrick, orgy = by * kBrick, orgz = bz * kBrick;
        for (int k = tid; k < 8 * kAccVox / 4; k += kAccThreads)
            reinterpret_cast<uint4*>(&acc[0][0])[k] = make_uint4(0u, 0u, 0u, 0u);
        for (int eb = e0; eb < e1; eb += kStage) {
            const int nbatch = min(kStage, e1 - eb);
            if (eb != e0) __syncthreads();       // the previous batch is done with
            if (tid < nbatch) {
                const int i = entries[eb + tid];
                const int4 pb = pbase[i];
                const float4 fr = pfrac[i], nr = pnrm[i];
                unsigned pk;
                if (WEIGHTED) {
                    // corner of the 4^3 stencil relative to the brick: -3 .. 7 per axis
                    pk = (unsigned)(pb.x - 1 - orgx + 8) | (unsigned)(pb.y - 1 - orgy + 8) << 12 |
                         (unsigned)(pb.z - 1 - orgz + 8) << 24;
                    // X - p(q) = (t - q) h with t - q = frac + 1 - offset
                    s_frac[tid] = make_float4(fr.x + 1.0f, fr.y + 1.0f, fr.z + 1.0f, fr.w);
                } else {
                    // the nearest node: inside the brick
                    pk = (unsigned)(pb.x + ((pb.w >> 1) & 1) - orgx) | (unsigned)(pb.y + ((pb.w >> 2) & 1) - orgy) << 3 |
                         (unsigned)(pb.z + ((pb.w >> 3) & 1) - orgz) << 6;
                }
                s_nrm[tid] = make_float4(nr.x, nr.y, nr.z, __uint_as_float(pk));
            }
            __syncthreads();
            if (WEIGHTED) {
                for (int p = warp; p < nbatch; p += kAccThreads / 32) {
                    const float4 nr = s_nrm[p], fr = s_frac[p];
                    const unsigned pk = __float_as_uint(nr.w), q = pk + lane_off;
                    const bool in_xy = (q & 0x18018u) == 0x08008u;
                    const int zc = (int)(pk >> 24) - 8;                 // first stencil plane, warp-uniform
                    const int z1 = min(3, 7 - zc);                      // last one in the brick
                    const float dx = (fr.x - fox) * g.hf[0];
                    const float dy = (fr.y - foy) * g.hf[1];
                    const float rxy = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
                    const int lxy = (int)((q & 7u) | ((q >> 9) & 0x38u));
                    for (int zb = max(0, -zc); zb <= z1; zb += 2) {
                        const int oz = zb + (lane >> 4);
                        if (!in_xy || oz > z1) continue;
                        const float dz = (fr.z - (float)oz) * g.hf[2];
                        const float r2 = __fmaf_rn(dz, dz, rxy);
                        const float e1v = expf(-r2 * g.inv_s1sq) * fr.w;   // sigma1 * g1 * W
                        const float e2v = expf(-r2 * g.inv_s2sq) * fr.w;   // sigma2 * g2 * W
                        const int li = lxy + kPlane * (zc + oz);
                        const float val[4] = {e1v * nr.x, e1v * nr.y, e1v * nr.z, e2v};
                        if (fast) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                int hi, lo;
                                fix40_split(val[c], hi, lo);
                                atomicAdd(reinterpret_cast<int*>(&acc[c][li]), hi);
                                atomicAdd(reinterpret_cast<int*>(&acc[4 + c][li]), lo);
                            }
                        } else {
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                atomicAdd(&acc64[c * kAccVox + li], (unsigned long long)fix40(val[c]));
                        }
                    }
                }
            } else {
                for (int p = tid; p < nbatch; p += kAccThreads) {
                    const float4 nr = s_nrm[p];
                    const int li = acc_of((int)__float_as_uint(nr.w));
                    const float val[3] = {nr.x, nr.y, nr.z};
                    if (fast) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            int hi, lo;
                            fix40_split(val[c], hi, lo);
                            atomicAdd(reinterpret_cast<int*>(&acc[c][li]), hi);
                            atomicAdd(reinterpret_cast<int*>(&acc[4 + c][li]), lo);
                        }
                        atomicAdd(reinterpret_cast<int*>(&acc[3][li]), 1 << 20);   // count: 2^40 = 2^20 * 2^20
                    } else {
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            atomicAdd(&acc64[c * kAccVox + li], (unsigned long long)fix40(val[c]));
                        atomicAdd(&acc64[3 * kAccVox + li], 1ull << 40);
                    }
                }
            }
        }
        __syncthreads();
        const int next = s_next;
        float* out = vpool + (size_t)s * 3 * kBrickVox;
        auto own_sums = [&](int a, long long (&u)[4]) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                u[c] = fast ? (long long)(int)acc[c][a] * (1ll << 20) + (long long)(int)acc[4 + c][a]
                            : (long long)acc64[c * kAccVox + a];
        };
        bool write = true;
        unsigned long long* gacc = nullptr;
        if (heavy) {
            // add this chunk's exact sums to the brick's global accumulator
            const int h = heavy_idx[s], nchunks = unit_off[s + 1] - unit_off[s];
            gacc = heavy_acc + (size_t)h * 4 * kBrickVox;
            for (int li = tid; li < kBrickVox; li += kAccThreads) {
                long long u[4];
                own_sums(acc_of(li), u);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (u[c] != 0) atomicAdd(&gacc[c * kBrickVox + li], (unsigned long long)u[c]);
            }
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                s_last = atomicAdd(&heavy_done[h], 1) == nchunks - 1;
                if (s_last) heavy_done[h] = 0;                          // cleared for the next frame
            }
            __syncthreads();
            write = s_last;                                             // block-uniform
            __threadfence();
        }
        if (write) {
            for (int li = tid; li < kBrickVox; li += kAccThreads) {
                long long u[4];
                if (gacc) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        u[c] = (long long)__ldcg(&gacc[c * kBrickVox + li]);
                        gacc[c * kBrickVox + li] = 0ull;                // cleared for the next frame
                    }
                } else {
                    own_sums(acc_of(li), u);
                }
                if (u[3] > 0) {
                    // exact integer sums, one float32 quotient per voxel
                    const float sc = g.v_scale_f / fix_to_float(u[3]);
                    out[li] = fix_to_float(u[0]) * sc;
                    out[kBrickVox + li] = fix_to_float(u[1]) * sc;
                    out[2 * kBrickVox + li] = fix_to_float(u[2]) * sc;
                } else {
                    out[li] = 0.f;
                    out[kBrickVox + li] = 0.f;
                    out[2 * kBrickVox + li] = 0.f;
                }
            }
        }
        unit = next;
        __syncthreads();                        // accumulators and s_next are free again
    }
}

__global__ void k_dense_V(GridDev g, const int* __restrict__ slot, const float* __restrict__ vpool, int64_t M,
                          float* out) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= M) return;
    const int x = (int)(q % g.n[0]);
    const int y = (int)((q / g.n[0]) % g.n[1]);
    const int z = (int)(q / ((int64_t)g.n[0] * g.n[1]));
    const int s = slot[(x >> 3) + g.nb[0] * ((y >> 3) + g.nb[1] * (z >> 3))];
    const int li = (x & 7) + 8 * ((y & 7) + 8 * (z & 7));
#pragma unroll
    for (int c = 0; c < 3; ++c)
        out[c * M + q] = s >= 0 ? vpool[(size_t)s * 3 * kBrickVox + c * kBrickVox + li] : 0.f;
}

__global__ void k_load_dense_V(GridDev g, const float* __restrict__ V, int64_t M, int* slot,
                               float* vpool) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= M) return;
    const int x = (int)(q % g.n[0]);
    const int y = (int)((q / g.n[0]) % g.n[1]);
    const int z = (int)(q / ((int64_t)g.n[0] * g.n[1]));
    const int b = (x >> 3) + g.nb[0] * ((y >> 3) + g.nb[1] * (z >> 3));
    const int li = (x & 7) + 8 * ((y & 7) + 8 * (z & 7));
    if (li == 0) slot[b] = b;
#pragma unroll
    for (int c = 0; c < 3; ++c) vpool[(size_t)b * 3 * kBrickVox + c * kBrickVox + li] = V[c * M + q];
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_ingest(ftr_ctx* c, const float* pts, const float* nrm, const float* w, int64_t n,
                          const int* n_dev) {
    if (n == 0) return cudaSuccess;
    if (cudaError_t e = cudaGetLastError()) return e;    // see launch_ingest_sets
    // small CTAs spread the few float64 operations per point over every SM; with
    // the count on the device (n = every depth pixel) they stride over it: a CTA
    // per 32 pixels ran 40,704 CTAs for 65,000 points, 24 us
    const unsigned blocks = n_dev ? (unsigned)min((int64_t)kSms * 32, (int64_t)blocks_for(n, 32)) : blocks_for(n, 32);
    launch_pdl(k_ingest, blocks, 32, 0, c->stream, pts, nrm, w, n, c->n_pts, c->g, c->pts.base, c->pts.frac,
                                                       c->pts.nrm, c->d_dropped, c->d_wild, c->d_npts, n_dev,
                                                       c->d_brick_cnt);
    c->launches++;
    return cudaGetLastError();
}

// The ingest counts its points into their bricks, which a second call would do
// again.  So an error that the application left on the thread, which ends the call,
// is looked for before the launch and not only behind it.
cudaError_t launch_ingest_sets(ftr_ctx* c, const IngestSets& S) {
    const int64_t n = S.off[S.k];
    if (n == 0) return cudaSuccess;
    if (cudaError_t e = cudaGetLastError()) return e;
    launch_pdl(k_ingest_sets, blocks_for(n, 32), 32, 0, c->stream, S, c->g, c->pts.base, c->pts.frac, c->pts.nrm,
               c->d_dropped, c->d_wild, c->d_npts, c->d_brick_cnt);
    c->launches++;
    return cudaGetLastError();
}

// The binning adds to the unit counts and the accumulation clears them for the
// next frame.  A solve that fails between the two (every launch reports errors
// of the thread, also ones the application left behind) leaves them standing:
// a frame binned on top of them would place its units at twice their number,
// past d_units where most bricks are touched.
cudaError_t clear_classes(ftr_ctx* c) {
    if (!c->class_dirty) return cudaSuccess;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(c->stream, &cs);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->d_meta + kMetaClasses, 0, sizeof(int) * 2 * kSizeClasses, c->stream);
    // a captured memset has not run yet: the flag stays for the next call
    if (e == cudaSuccess && cs == cudaStreamCaptureStatusNone) c->class_dirty = false;
    return e;
}

cudaError_t launch_splat(ftr_ctx* c) {
    cudaError_t e;
    const bool dirty = c->class_dirty;
    c->class_dirty = true;                       // until the accumulation is enqueued
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (sms <= 0) sms = kSms;
    prof_begin(c, ST_SPLAT_BIN);
    // the per-brick point counts were taken by the ingest
    const int ntiles = (c->n_bricks + kTile - 1) / kTile;
    launch_pdl(k_brick_tile_sums, ntiles, kScanT, 0, c->stream, c->d_brick_cnt, c->n_bricks, c->d_tile, c->d_meta);
    launch_pdl(k_brick_tile_write, ntiles, kScanT, 0, c->stream, c->d_brick_cnt, c->n_bricks, c->g.nb[0], c->g.nb[0] * c->g.nb[1],
               c->d_tile, ntiles, c->d_brick_cursor, c->d_brick_slot, c->d_meta,
               c->d_unit_off, c->d_heavy_idx, c->d_units);
    c->launches += 2;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_pdl(k_brick_fill, sms * 2, 256, 0, c->stream, c->pts.base, c->d_npts, c->g, c->d_brick_cursor, c->d_entries);
    c->launches++;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    prof_end(c, ST_SPLAT_BIN);
    prof_begin(c, ST_SPLAT_ACC);
    const int grid = sms * 6;
    launch_pdl(c->g.mode == FTR_SPLAT_WEIGHTED ? k_splat_accum<true> : k_splat_accum<false>, grid, kAccThreads, 0,
               c->stream, c->g, c->d_meta, c->d_units, c->d_entries, c->pts.base, c->pts.frac, c->pts.nrm, c->d_wild,
               c->d_vpool, c->d_unit_off, c->d_heavy_idx, c->d_heavy_acc, c->d_heavy_done);
    c->launches++;
    prof_end(c, ST_SPLAT_ACC);
    if ((e = cudaGetLastError()) == cudaSuccess) c->class_dirty = dirty;
    return e;
}

cudaError_t launch_load_dense_V(ftr_ctx* c, const float* V_dev) {
    k_load_dense_V<<<blocks_for(c->M, 256), 256, 0, c->stream>>>(c->g, V_dev, c->M, c->d_brick_slot, c->d_vpool);
    c->launches++;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int meta[4] = {c->n_bricks, 0, 0, c->g.nb[2] - 1};
    if ((e = cudaMemsetAsync(c->d_meta + kMetaRows, 0xff, sizeof(int) * (kMetaClasses - kMetaRows), c->stream)) != cudaSuccess)
        return e;
    return cudaMemcpyAsync(c->d_meta, meta, sizeof(meta), cudaMemcpyHostToDevice, c->stream);
}

cudaError_t launch_dense_V(ftr_ctx* c, float* out_dev) {
    k_dense_V<<<blocks_for(c->M, 256), 256, 0, c->stream>>>(c->g, c->d_brick_slot, c->d_vpool, c->M, out_dev);
    c->launches++;
    return cudaGetLastError();
}

}  // namespace ftr

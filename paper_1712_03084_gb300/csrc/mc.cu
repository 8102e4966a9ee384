// Marching cubes on A at level L (Sec. III-B, [35]), scan-compacted.
//
// Corner bit = 1 iff A >= L with A promoted to float64.  Because A is float32,
// that is the same as A >= Lf with Lf = L rounded up to float32, so the
// kernels compare in float32 and still take the float64 decision.  A node owns
// the grid edges toward +x, +y, +z; an edge carries a vertex when its two bits
// differ.  Vertex ids are the rank of (node, axis) in linear node order and
// triangles follow cell order then table order, so the mesh does not depend
// on scheduling.
//
// The inside bits are computed once (one warp per grid row, one ballot per
// 32 nodes: 1 bit per node, 2 MB at 256^3) and both passes below work on
// 32-node words: a thread takes word w of row (y, z) and the same word of
// the rows (y+1, z), (y, z+1), (y+1, z+1); XORs give the crossing edges
// toward +x, +y, +z and AND/OR of the eight corner masks the cells whose
// corners differ (exactly the cells with triangles).  Launches:
//   bits   a class per grid row (outside, inside, mixed) and the inside bits
//          of the mixed rows
//   count  per tile of (row, word) threads: active nodes (owning a vertex
//          or lower corner of a cell with triangles), vertices, triangles;
//          also summed per group of 256 tiles
//   emit   per tile with an active node: its offset from the group and tile
//          sums before it, a CTA scan of its counts, per active node in x
//          order one 16-byte record (node, edge bits | class << 8, first
//          vertex, first triangle), and per word with active nodes its first
//          record index and active mask
//   tris   one thread per active node: the vertices of its crossing edges
//          (t = (L - A0)/(A1 - A0), normal -grad A by central differences,
//          one-sided at the border, lerped), then its triangles' corners
//          from the case table; the record of an edge's owner node is its
//          word's first record plus the active nodes before it in the word.
#include <cuda_runtime.h>
#include <math.h>

#include "ftr_internal.h"

namespace ftr {
namespace {

__constant__ int c_ntri[256];
__constant__ signed char c_tri[256][kMaxTrisPerCase][3];


struct NodeInfo {
    int flags;     // bit a: edge toward +a crosses
    int cls;       // cube class, 0 if the node is not a cell's lower corner
};

__device__ __forceinline__ NodeInfo classify_node(const float* __restrict__ A, int64_t n, int x, int y, int z,
                                                  const GridDev& g, float L) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int64_t sy = nx, sz = (int64_t)nx * ny;
    const bool hx = x < nx - 1, hy = y < ny - 1, hz = z < nz - 1;
    const int b0 = A[n] >= L;
    NodeInfo r;
    r.flags = 0;
    r.cls = 0;
    const int bx = hx ? (A[n + 1] >= L) : b0;
    const int by = hy ? (A[n + sy] >= L) : b0;
    const int bz = hz ? (A[n + sz] >= L) : b0;
    r.flags = (bx != b0) | ((by != b0) << 1) | ((bz != b0) << 2);
    if (hx && hy && hz) {
        const int bxy = A[n + 1 + sy] >= L;
        const int bxz = A[n + 1 + sz] >= L;
        const int byz = A[n + sy + sz] >= L;
        const int bxyz = A[n + 1 + sy + sz] >= L;
        r.cls = b0 | (bx << 1) | (by << 2) | (bxy << 3) | (bz << 4) | (bxz << 5) | (byz << 6) | (bxyz << 7);
    }
    return r;
}

__device__ __forceinline__ int ntri_of(int cls) { return (cls == 0 || cls == 255) ? 0 : c_ntri[cls]; }

// ---------------------------------------------------------------- bit masks
// The inside bits (A >= L) of every node, 32 per word: word w of grid row r
// (y + n_y z) holds x = 32 w .. 32 w + 31 (bit i = node 32 w + i; zero past
// n_x); rows are `wp` words apart (wp = the words per row rounded up to a
// power of two).  Per row a class: every node outside (0), every node inside
// (1) or mixed (2).  Most rows of a grid are not mixed; their words are neither
// computed nor (unless `all`) written, and the passes below take them from the
// class.
// rowmm (nullable): per row the minimum and maximum of A, from which a row
// whose maximum is below the level, or whose minimum is at or above it, gets
// its class without reading A (the same bits: every node of the row decides
// alike); else the class comes from the words.
// It also zeroes `zero[0 .. nzero)` (the group sums of k_mc_count_tiles).
constexpr int kOutside = 0, kInside = 1, kMixed = 2;
constexpr int kBitRows = 4;          // grid rows per warp: a quarter of the CTAs for rows that end at their class

// Nodes of word w that exist.
__device__ __forceinline__ unsigned word_valid(int nx, int w) {
    const int left = nx - 32 * w;
    return left >= 32 ? 0xffffffffu : (left <= 0 ? 0u : (1u << left) - 1u);
}

__global__ void __launch_bounds__(kMcThreads) k_mc_bits(GridDev g, const float* __restrict__ A,
                                                        const float* __restrict__ levelf, unsigned* __restrict__ bits,
                                                        unsigned char* __restrict__ cls, int nrows, int wp,
                                                        int* __restrict__ zero, int nzero,
                                                        const float2* __restrict__ rowmm, int all) {
    pdl_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nzero; i += gridDim.x * blockDim.x) zero[i] = 0;
    const int lane = threadIdx.x & 31;
    const float L = levelf[0];
    const int nx = g.n[0];
    const int nw = (nx + 31) >> 5;
    const int row0 = (blockIdx.x * (kMcThreads / 32) + (threadIdx.x >> 5)) * kBitRows;
    if (row0 >= nrows) return;                  // warp-uniform; nrows is a multiple of kBitRows
    int c = kMixed;
    if (rowmm && lane < kBitRows) {
        const float2 mm = rowmm[row0 + lane];
        c = mm.y < L ? kOutside : (mm.x >= L ? kInside : kMixed);   // mixed for NaN bounds
    }
    const unsigned mixed = rowmm ? __ballot_sync(0xffffffffu, lane < kBitRows && c == kMixed) : (1u << kBitRows) - 1u;
    for (unsigned m = mixed; m; m &= m - 1) {
        const int r = __ffs(m) - 1;
        const float* a = A + (int64_t)(row0 + r) * nx;
        unsigned mine = 0u;
        // up to 8 words per batch: all loads are issued before the first ballot
        for (int w0 = 0; w0 < nw; w0 += 8) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int x = 32 * (w0 + k) + lane;
                v[k] = x < nx ? a[x] : -INFINITY;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const unsigned b = __ballot_sync(0xffffffffu, v[k] >= L);
                if (lane == w0 + k) mine = b;
            }
        }
        const unsigned valid = word_valid(nx, lane);
        mine &= valid;
        if (!rowmm) {
            const bool some = __any_sync(0xffffffffu, mine != 0u), every = __all_sync(0xffffffffu, mine == valid);
            if (lane == r) c = !some ? kOutside : (every ? kInside : kMixed);
        }
        if (lane < wp) bits[(int64_t)(row0 + r) * wp + lane] = mine;
    }
    if (lane < kBitRows) cls[row0 + lane] = (unsigned char)c;
    if (all && rowmm) {
        for (int r = 0; r < kBitRows; ++r) {
            const int rc = __shfl_sync(0xffffffffu, c, r);
            if (rc != kMixed && lane < wp)
                bits[(int64_t)(row0 + r) * wp + lane] = rc == kInside ? word_valid(nx, lane) : 0u;
        }
    }
}

// Per (row, word): the masks of the nodes of word w that own a crossing
// edge toward +x, +y, +z, and that are the lower corner of a cell whose
// corners are not all on one side ("mixed": exactly the cells with
// triangles).  Nodes with any of the four are the row's active nodes.
struct WordMasks {
    unsigned ex, ey, ez, mixed;
    unsigned c[8];   // corner bits of the cells whose lower corner is in the word
};

// Classes of the row, of its +y, +z and +y+z neighbours (the row's own where
// the grid ends), and whether a surface can pass between them.
struct RowClasses {
    int c00, c10, c01, c11;
    bool live;
};

__device__ __forceinline__ RowClasses row_classes(const unsigned char* __restrict__ cls, int row, bool hy, bool hz,
                                                  int ny) {
    RowClasses r;
    r.c00 = cls[row];
    r.c10 = hy ? cls[row + 1] : r.c00;
    r.c01 = hz ? cls[row + ny] : r.c00;
    r.c11 = hy && hz ? cls[row + ny + 1] : r.c00;
    const int any = r.c00 | r.c10 | r.c01 | r.c11;
    r.live = any > kInside || (any != r.c00 || r.c00 != r.c10 || r.c00 != r.c01 || r.c00 != r.c11);
    return r;
}

__device__ __forceinline__ WordMasks word_masks(const unsigned* __restrict__ bits, const RowClasses& rc, int row, int w,
                                                int nw, int wp, int x_count, bool hy, bool hz, int ny) {
    const int64_t r00 = (int64_t)row * wp, r10 = r00 + wp, r01 = r00 + (int64_t)ny * wp, r11 = r01 + wp;
    const bool more = w + 1 < nw;
    // nodes of the word (and of the next) that exist, and those with a +x neighbour
    const int base = 32 * w;
    const unsigned valid = word_valid(x_count, w), nvalid = word_valid(x_count, w + 1);
    auto word = [&](int c, int64_t r) { return c == kMixed ? bits[r + w] : (c == kInside ? valid : 0u); };
    auto next = [&](int c, int64_t r) { return !more ? 0u : (c == kMixed ? bits[r + w + 1] : (c == kInside ? nvalid : 0u)); };
    const unsigned b00 = word(rc.c00, r00), n00 = next(rc.c00, r00);
    const unsigned b10 = hy ? word(rc.c10, r10) : 0u, n10 = hy ? next(rc.c10, r10) : 0u;
    const unsigned b01 = hz ? word(rc.c01, r01) : 0u, n01 = hz ? next(rc.c01, r01) : 0u;
    const unsigned b11 = (hy && hz) ? word(rc.c11, r11) : 0u, n11 = (hy && hz) ? next(rc.c11, r11) : 0u;
    const unsigned vx = x_count - 1 - base >= 32 ? 0xffffffffu
                        : (x_count - 1 - base <= 0 ? 0u : ((1u << (x_count - 1 - base)) - 1u));
    WordMasks m;
    m.c[0] = b00;
    m.c[1] = (b00 >> 1) | (n00 << 31);
    m.c[2] = b10;
    m.c[3] = (b10 >> 1) | (n10 << 31);
    m.c[4] = b01;
    m.c[5] = (b01 >> 1) | (n01 << 31);
    m.c[6] = b11;
    m.c[7] = (b11 >> 1) | (n11 << 31);
    m.ex = (m.c[0] ^ m.c[1]) & vx;
    m.ey = hy ? ((b00 ^ b10) & valid) : 0u;
    m.ez = hz ? ((b00 ^ b01) & valid) : 0u;
    unsigned all = 0xffffffffu, any = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        all &= m.c[k];
        any |= m.c[k];
    }
    m.mixed = (hy && hz) ? ((any & ~all) & vx) : 0u;
    return m;
}

__device__ __forceinline__ int cell_class(const WordMasks& m, int i) {
    int cls = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) cls |= (int)((m.c[k] >> i) & 1u) << k;
    return cls;
}

// Block-wide exclusive scan of 3 ints (T threads); returns totals.
template <int T>
__device__ __forceinline__ int3 block_scan3(int3 v, int3& total, int3* sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int3 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, inc.x, o);
        const int b = __shfl_up_sync(0xffffffffu, inc.y, o);
        const int c = __shfl_up_sync(0xffffffffu, inc.z, o);
        if (lane >= o) {
            inc.x += a;
            inc.y += b;
            inc.z += c;
        }
    }
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int3 w = lane < T / 32 ? sh[lane] : make_int3(0, 0, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, w.x, o);
            const int b = __shfl_up_sync(0xffffffffu, w.y, o);
            const int c = __shfl_up_sync(0xffffffffu, w.z, o);
            if (lane >= o) {
                w.x += a;
                w.y += b;
                w.z += c;
            }
        }
        if (lane < T / 32) sh[lane] = w;
    }
    __syncthreads();
    const int3 before = wid ? sh[wid - 1] : make_int3(0, 0, 0);
    total = sh[T / 32 - 1];
    __syncthreads();
    return make_int3(before.x + inc.x - v.x, before.y + inc.y - v.y, before.z + inc.z - v.z);
}

// ------------------------------------------------- tiles: count, then emit
// Both kernels run over the (row, word) threads in node order in the same
// tiles of T threads (the context's marching-cubes tile size: 128, 256 or
// 512; the mesh does not depend on it).  The count kernel writes each tile's sums (active
// nodes, vertices, triangles) and adds them into its group's sums (256 tiles
// per group; integer atomics, so the order does not matter).  The emit
// kernel's tile gets its offset from the groups before it and the tiles
// before it in its group (at most 255 + a few loads, spread over the CTA),
// scans its own counts, and writes its node records.
//
// Tile state (agg) and group sums (sup, zeroed by k_mc_bits) as int4: active
// nodes, vertices, triangles, unused.
struct WordCounts {
    WordMasks m;
    unsigned act;
    int3 c;
};

__device__ __forceinline__ WordCounts word_counts(const GridDev& g, const unsigned* __restrict__ bits,
                                                  const RowClasses& rc, int row, int w, int wp,
                                                  const unsigned char* s_ntri) {
    WordCounts r;
    r.act = 0u;
    r.c = make_int3(0, 0, 0);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int nw = (nx + 31) >> 5;
    if (rc.live && w < nw) {
        const int y = row % ny, z = row / ny;
        r.m = word_masks(bits, rc, row, w, nw, wp, nx, y < ny - 1, z < nz - 1, ny);
        r.act = r.m.ex | r.m.ey | r.m.ez | r.m.mixed;
        r.c.x = __popc(r.act);
        r.c.y = __popc(r.m.ex) + __popc(r.m.ey) + __popc(r.m.ez);
        unsigned mm = r.m.mixed;
        while (mm) {
            const int i = __ffs(mm) - 1;
            mm &= mm - 1;
            r.c.z += s_ntri[cell_class(r.m, i)];
        }
    }
    return r;
}

constexpr int kMcGroup = 256;     // tiles per group sum

// A tile whose rows and their neighbours are all on one side (four fifths of a
// body's grid) ends after the row classes; 9216 tiles of a 384^3 frame: 33 us
// when every tile read its words and scanned its counts.
template <int T>
__global__ void __launch_bounds__(T) k_mc_count_tiles(GridDev g, const unsigned* __restrict__ bits,
                                                               const unsigned char* __restrict__ cls, int nrows, int wp,
                                                               int4* __restrict__ agg, int* __restrict__ sup) {
    pdl_wait();
    __shared__ unsigned char s_ntri[256];
    __shared__ int s_sum[3];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int row = (int)(t / wp), w = (int)(t % wp);
    RowClasses rc;
    rc.live = false;
    if (row < nrows) rc = row_classes(cls, row, row % g.n[1] < g.n[1] - 1, row / g.n[1] < g.n[2] - 1, g.n[1]);
    if (!__syncthreads_or(rc.live)) {
        if (threadIdx.x == 0) agg[blockIdx.x] = make_int4(0, 0, 0, 0);
        return;
    }
    for (int k = threadIdx.x; k < 256; k += blockDim.x) s_ntri[k] = (unsigned char)c_ntri[k];
    if (threadIdx.x < 3) s_sum[threadIdx.x] = 0;
    __syncthreads();
    const WordCounts wc = word_counts(g, bits, rc, row, w, wp, s_ntri);
    const int3 sum = make_int3(__reduce_add_sync(0xffffffffu, wc.c.x), __reduce_add_sync(0xffffffffu, wc.c.y),
                               __reduce_add_sync(0xffffffffu, wc.c.z));
    if ((threadIdx.x & 31) == 0 && (sum.x | sum.y | sum.z)) {
        atomicAdd(&s_sum[0], sum.x);
        atomicAdd(&s_sum[1], sum.y);
        atomicAdd(&s_sum[2], sum.z);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int3 tot = make_int3(s_sum[0], s_sum[1], s_sum[2]);
        agg[blockIdx.x] = make_int4(tot.x, tot.y, tot.z, 0);
        int* s = sup + 4 * (blockIdx.x / kMcGroup);
        if (tot.x) atomicAdd(&s[0], tot.x);
        if (tot.y) atomicAdd(&s[1], tot.y);
        if (tot.z) atomicAdd(&s[2], tot.z);
    }
}

template <int T>
__global__ void __launch_bounds__(T) k_mc_emit_tiles(GridDev g, const unsigned* __restrict__ bits,
                                                              const unsigned char* __restrict__ cls, int nrows, int wp,
                                                              int ntiles, const int4* __restrict__ agg,
                                                              const int4* __restrict__ sup, int* __restrict__ totals,
                                                              int4* __restrict__ nodes, int cap_nodes,
                                                              int2* __restrict__ wordinfo,
                                                              int* __restrict__ host_totals) {
    pdl_wait();
    __shared__ unsigned char s_ntri[256];
    __shared__ int3 sh[T / 32];
    const int tile = blockIdx.x, grp = tile / kMcGroup;
    // a tile the count found empty (most of the grid) has nothing to write; the
    // last one reports the totals
    const int4 mine = agg[tile];
    const bool empty = (mine.x | mine.y | mine.z) == 0;
    if (empty && tile != ntiles - 1) return;
    for (int k = threadIdx.x; k < 256; k += blockDim.x) s_ntri[k] = (unsigned char)c_ntri[k];
    // the sums of every tile before this one: whole groups, then this group's tiles
    int3 pre = make_int3(0, 0, 0);
    for (int k = threadIdx.x; k < grp; k += blockDim.x) {
        const int4 v = sup[k];
        pre.x += v.x;
        pre.y += v.y;
        pre.z += v.z;
    }
    for (int k = grp * kMcGroup + threadIdx.x; k < tile; k += blockDim.x) {
        const int4 v = agg[k];
        pre.x += v.x;
        pre.y += v.y;
        pre.z += v.z;
    }
    __syncthreads();
    int3 base;
    block_scan3<T>(pre, base, sh);
    if (tile == ntiles - 1 && threadIdx.x == 0) {
        // totals for the kernels that follow and, in page-locked memory, for the host
        totals[0] = host_totals[0] = base.x + mine.x;
        totals[1] = host_totals[1] = base.y + mine.y;
        totals[2] = host_totals[2] = base.z + mine.z;
    }
    if (empty) return;
    const int64_t t = (int64_t)tile * blockDim.x + threadIdx.x;
    const int row = (int)(t / wp), w = (int)(t % wp);
    RowClasses rc;
    rc.live = false;
    if (row < nrows) rc = row_classes(cls, row, row % g.n[1] < g.n[1] - 1, row / g.n[1] < g.n[2] - 1, g.n[1]);
    const WordCounts wc = word_counts(g, bits, rc, row, w, wp, s_ntri);
    int3 tot;
    const int3 ex = block_scan3<T>(wc.c, tot, sh);
    int ja = base.x + ex.x, jv = base.y + ex.y, jt = base.z + ex.z;
    // the word's first record and its active nodes: the triangle pass finds
    // a corner's owner record from these without scanning the row
    if (wc.act) wordinfo[t] = make_int2(ja, (int)wc.act);
    const int64_t rowbase = (int64_t)row * g.n[0];
    unsigned rem = wc.act;
    while (rem) {
        const int i = __ffs(rem) - 1;
        rem &= rem - 1;
        const int flags = (int)((wc.m.ex >> i) & 1u) | ((int)((wc.m.ey >> i) & 1u) << 1) |
                          ((int)((wc.m.ez >> i) & 1u) << 2);
        const int cls = ((wc.m.mixed >> i) & 1u) ? cell_class(wc.m, i) : 0;
        if (ja < cap_nodes) nodes[ja] = make_int4((int)(rowbase + 32 * w + i), flags | (cls << 8), jv, jt);
        ++ja;
        jv += __popc(flags);
        jt += cls ? s_ntri[cls] : 0;
    }
}

// Vertices on the crossing edges of node n: t = (L - A0) / (A1 - A0) and the
// position p(q) + t h_a e_a, in float32 (no decision depends on them; the
// error is a few float32 ulps of the coordinates), normal = -grad A lerped
// (central differences, one-sided at the border).  All reads (the node's six
// neighbours, five more per crossing edge) are issued before the first use:
// edge by edge they were a chain of round trips.
__device__ __forceinline__ void emit_vertices(const GridDev& g, const float* __restrict__ A, float Ln,
                                              int64_t n, const int q[3], int flags, int vi, int cap_v,
                                              float* __restrict__ verts, float* __restrict__ vnrm) {
    const int nn[3] = {g.n[0], g.n[1], g.n[2]};
    const int64_t st[3] = {1, (int64_t)g.n[0], (int64_t)g.n[0] * g.n[1]};
    const float a0 = A[n];
    float fw[3], bw[3];                     // neighbours of the node; itself where the grid ends
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        fw[c] = q[c] < nn[c] - 1 ? A[n + st[c]] : a0;
        bw[c] = q[c] > 0 ? A[n - st[c]] : a0;
    }
    float hi[3][3], lo[3][3];               // per edge: the neighbours of its far node
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!((flags >> a) & 1)) continue;
        const int64_t n1 = n + st[a];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int qc = q[c] + (c == a ? 1 : 0);
            hi[a][c] = qc < nn[c] - 1 ? A[n1 + st[c]] : fw[a];
            lo[a][c] = c == a ? a0 : (qc > 0 ? A[n1 - st[c]] : fw[a]);
        }
    }
    float g0[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
        g0[c] = (fw[c] - bw[c]) * (q[c] == 0 || q[c] == nn[c] - 1 ? g.inv_hf[c] : 0.5f * g.inv_hf[c]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!((flags >> a) & 1)) continue;
        const float tt = (Ln - a0) / (fw[a] - a0);
        float p[3], nv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int q1 = q[c] + (c == a ? 1 : 0);
            const float g1 = (hi[a][c] - lo[a][c]) * (q1 == 0 || q1 == nn[c] - 1 ? g.inv_hf[c] : 0.5f * g.inv_hf[c]);
            const float qc = (float)q[c] + 0.5f + (c == a ? tt : 0.0f);
            p[c] = fmaf(qc, g.hf[c], g.bminf[c]);
            nv[c] = -__fmaf_rn(1.0f - tt, g0[c], __fmul_rn(tt, g1));
        }
        const float len2 = __fmaf_rn(nv[2], nv[2], __fmaf_rn(nv[0], nv[0], __fmul_rn(nv[1], nv[1])));
        const float inv = len2 > 0.f ? rsqrtf(len2) : 0.f;
        if (vi >= cap_v) return;   // buffers too small: the host grows them and runs again
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            verts[3 * (int64_t)vi + c] = p[c];
            vnrm[3 * (int64_t)vi + c] = nv[c] * inv;
        }
        ++vi;
    }
}

constexpr int kTriThreads = 256;

// Triangles of a node's cell.  The owner of a cube edge's vertex is the node at
// the edge's lower end: this node or a neighbour toward +x, +y, +z.  It is
// active (it owns the crossing edge), so its word was written by the emit pass:
// its record index is the word's first record plus the active nodes before it
// in the word.  The six neighbours' records are looked up together (one round
// trip for the words, one for the records; corner by corner it was two per
// corner), the twelve edges' vertex ids go to this thread's column of s_edge
// and the case table picks from them.
__device__ __forceinline__ void tris_of_node(const GridDev& g, const int4* __restrict__ nodes, const int4 rec,
                                             const int2* __restrict__ wordinfo, int wp, int n_nodes,
                                             int32_t* __restrict__ tris, int (*s_edge)[kTriThreads]) {
    const int cls = rec.y >> 8;
    const int nt = ntri_of(cls);
    if (nt == 0) return;
    const int nx = g.n[0], ny = g.n[1];
    const int row = rec.x / nx;
    const int x = rec.x - row * nx;
    // corner b of the cube at (b & 1, b >> 1 & 1, b >> 2 & 1); owner b is needed
    // when one of its edges toward +a inside the cube crosses
    int first[7], below[7];
    first[0] = rec.z;
    below[0] = rec.y;
    int2 wi[7];
    bool need[7];
#pragma unroll
    for (int b = 1; b < 7; ++b) {
        const int in = (cls >> b) & 1;
        need[b] = false;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (!((b >> a) & 1)) need[b] = need[b] || ((cls >> (b | (1 << a))) & 1) != in;
        if (need[b])
            wi[b] = wordinfo[(int64_t)(row + ((b >> 1) & 1) + ny * (b >> 2)) * wp + ((x + (b & 1)) >> 5)];
    }
#pragma unroll
    for (int b = 1; b < 7; ++b) {
        if (!need[b]) continue;
        const unsigned before = (unsigned)wi[b].y & ((1u << ((x + (b & 1)) & 31)) - 1u);
        // clamped: an inconsistent lookup gives a wrong index, never an access outside the records
        const int4 o = nodes[min(max(wi[b].x + __popc(before), 0), n_nodes - 1)];
        first[b] = o.z;
        below[b] = o.y;
    }
    const int tid = threadIdx.x;
    // edge 4 a + c_u + 2 c_v: from corner (c_u, c_v) on the two other axes toward +a
#pragma unroll
    for (int e = 0; e < 12; ++e) {
        const int a = e >> 2, cu = e & 1, cv = (e >> 1) & 1;
        const int b = a == 0 ? (cu << 1) | (cv << 2) : (a == 1 ? cu | (cv << 2) : cu | (cv << 1));
        if (((cls >> b) & 1) != ((cls >> (b | (1 << a))) & 1))
            s_edge[e][tid] = first[b] + __popc(below[b] & ((1 << a) - 1));
    }
    for (int k = 0; k < nt; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) tris[3 * (int64_t)(rec.w + k) + j] = s_edge[c_tri[cls][k][j]][tid];
}

// One thread per node record: the vertices on its crossing edges, then its
// triangles.
__global__ void __launch_bounds__(kTriThreads) k_mc_tris(GridDev g, const float* __restrict__ A,
                                                         const float* __restrict__ levelf,
                                                         const int4* __restrict__ nodes,
                                                         const int* __restrict__ totals, int cap_nodes, int cap_tris,
                                                         const int2* __restrict__ wordinfo, int wp,
                                                         int32_t* __restrict__ tris, float* __restrict__ verts,
                                                         float* __restrict__ vnrm, int cap_v) {
    pdl_wait();
    __shared__ int s_edge[12][kTriThreads];
    const int n_nodes = totals[0];
    if (n_nodes > cap_nodes || totals[2] > cap_tris) return;   // the host grows the buffers and runs again
    const float Ln = levelf[1];
    const int nx = g.n[0], ny = g.n[1];
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n_nodes; r += gridDim.x * blockDim.x) {
        const int4 rec = nodes[r];
        const int flags = rec.y & 7;
        if (flags) {
            const int row = rec.x / nx;
            const int q[3] = {rec.x - row * nx, row % ny, row / ny};
            emit_vertices(g, A, Ln, (int64_t)rec.x, q, flags, rec.z, cap_v, verts, vnrm);
        }
        tris_of_node(g, nodes, rec, wordinfo, wp, n_nodes, tris, s_edge);
    }
}

// n words from src to dst, 16 bytes at a time where both allow it.
__device__ __forceinline__ void copy_words(const uint32_t* __restrict__ src, uint32_t* __restrict__ dst, int64_t n) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
        const uint4* s = reinterpret_cast<const uint4*>(src);
        uint4* d = reinterpret_cast<uint4*>(dst);
        for (int64_t i = t; i < n / 4; i += step) d[i] = s[i];
        done = n / 4 * 4;
    }
    for (int64_t i = done + t; i < n; i += step) dst[i] = src[i];
}

// The mesh arrays into caller-owned device buffers: one launch where three
// device copies cost 2-3 us each.
__global__ void __launch_bounds__(256) k_mesh_copy(const float* __restrict__ v, const float* __restrict__ nrm,
                                                   const int32_t* __restrict__ tris, int64_t nv, int64_t nt,
                                                   float* vo, float* no, int32_t* to) {
    if (vo) copy_words(reinterpret_cast<const uint32_t*>(v), reinterpret_cast<uint32_t*>(vo), 3 * nv);
    if (no) copy_words(reinterpret_cast<const uint32_t*>(nrm), reinterpret_cast<uint32_t*>(no), 3 * nv);
    if (to) copy_words(reinterpret_cast<const uint32_t*>(tris), reinterpret_cast<uint32_t*>(to), 3 * nt);
}

__global__ void k_raise_flag(int* flag) { atomicExch(flag, 1); }

__global__ void k_mc_classes(GridDev g, const float* __restrict__ A, const float* __restrict__ levelf,
                             uint8_t* out) {
    const int cx = g.n[0] - 1, cy = g.n[1] - 1, cz = g.n[2] - 1;
    const int64_t ncell = (int64_t)cx * cy * cz;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ncell) return;
    const int z = (int)(i / ((int64_t)cx * cy));
    const int rem = (int)(i - (int64_t)z * cx * cy);
    const int y = rem / cx;
    const int x = rem - y * cx;
    const int64_t n = x + (int64_t)g.n[0] * (y + (int64_t)g.n[1] * z);
    out[i] = (uint8_t)classify_node(A, n, x, y, z, g, levelf[0]).cls;
}

}  // namespace

cudaError_t mc_init() {
    int32_t ntri[256];
    int32_t tris[256 * kMaxTrisPerCase * 3];
    mc_generate_table(ntri, tris);
    signed char t8[256][kMaxTrisPerCase][3];
    for (int c = 0; c < 256; ++c)
        for (int t = 0; t < kMaxTrisPerCase; ++t)
            for (int j = 0; j < 3; ++j) t8[c][t][j] = (signed char)tris[(c * kMaxTrisPerCase + t) * 3 + j];
    cudaError_t e = cudaMemcpyToSymbol(c_ntri, ntri, sizeof(ntri));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(c_tri, t8, sizeof(t8));
}

// Words per grid row of the inside bits, rounded up to a power of two.
static int mc_words(int nx) {
    const int nw = (nx + 31) / 32;
    int wp = 1;
    while (wp < nw) wp <<= 1;
    return wp;
}

// Tiles of T (row, word) threads (T = the context's marching-cubes tile size),
// and where the tile sums and the
// group sums sit in the per-row count buffer (3 x n_rows ints: room for both
// with up to 16 words per row, every supported grid).
static int mc_tiles(int nrows, int wp, int t) { return (int)(((int64_t)nrows * wp + t - 1) / t); }
static int mc_groups(int ntiles) { return (ntiles + kMcGroup - 1) / kMcGroup; }

// CTAs of the inside-bit pass: kBitRows rows per warp.  (A grid of one resident
// wave taking rows in a stride was as fast for one frame and 4-7 % slower
// when frames of several contexts overlap: short CTAs fill in around other
// kernels' CTAs.)
static unsigned mc_bits_grid(int nrows) {
    constexpr int per = kMcThreads / 32 * kBitRows;
    return (unsigned)((nrows + per - 1) / per);
}

cudaError_t launch_mc_bits(ftr_ctx* c) {
    const int nr = c->mc_blocks;
    launch_pdl(k_mc_bits, mc_bits_grid(nr), kMcThreads, 0, c->stream, c->g, c->d_A, c->d_levelf,
               c->d_mc_bits, c->d_mc_cls, nr, mc_words(c->g.n[0]), (int*)nullptr, 0,
               (const float2*)(c->rowmm_valid ? c->d_rowmm : nullptr), 1);
    c->launches++;
    return cudaGetLastError();
}

int mc_words_per_row(int nx) { return mc_words(nx); }

// A launch of the count or emit kernel instantiated for the tile size T.
template <template <int> class K, class... Args>
void launch_tiles(int t, int ntiles, cudaStream_t st, Args... args) {
    switch (t) {
        case 128: launch_pdl(K<128>::fn, ntiles, 128, 0, st, args...); break;
        case 512: launch_pdl(K<512>::fn, ntiles, 512, 0, st, args...); break;
        default: launch_pdl(K<256>::fn, ntiles, 256, 0, st, args...); break;
    }
}
template <int T> struct CountK { static constexpr auto fn = k_mc_count_tiles<T>; };
template <int T> struct EmitK { static constexpr auto fn = k_mc_emit_tiles<T>; };

bool mc_plan_valid(int tile, int tris_per_sm) {
    return (tile == 128 || tile == 256 || tile == 512) && tris_per_sm >= 1 && tris_per_sm <= 16;
}

cudaError_t launch_mc_count(ftr_ctx* c) {
    const int nr = c->mc_blocks;              // grid rows n_y n_z
    const int wp = mc_words(c->g.n[0]);
    const int ntiles = mc_tiles(nr, wp, c->mc_tile);
    if (4 * (ntiles + mc_groups(ntiles)) > 3 * nr) return cudaErrorInvalidValue;
    int4* agg = reinterpret_cast<int4*>(c->d_mc_blk);
    int* sup = c->d_mc_blk + 4 * ntiles;
    prof_begin(c, ST_MC_COUNT);
    launch_pdl(k_mc_bits, mc_bits_grid(nr), kMcThreads, 0, c->stream, c->g, c->d_A, c->d_levelf,
               c->d_mc_bits, c->d_mc_cls, nr, wp, sup, 4 * mc_groups(ntiles),
               (const float2*)(c->rowmm_valid ? c->d_rowmm : nullptr), 0);
    launch_tiles<CountK>(c->mc_tile, ntiles, c->stream, c->g, (const unsigned*)c->d_mc_bits,
                         (const unsigned char*)c->d_mc_cls, nr, wp, agg, sup);
    c->launches += 2;
    cudaError_t e = cudaGetLastError();
    prof_end(c, ST_MC_COUNT);
    return e;
}

// The node records, then the vertices and triangles.
cudaError_t launch_mc_emit(ftr_ctx* c) {
    const int nr = c->mc_blocks;
    const int wp = mc_words(c->g.n[0]);
    const int ntiles = mc_tiles(nr, wp, c->mc_tile);
    const int4* agg = reinterpret_cast<const int4*>(c->d_mc_blk);
    const int4* sup = reinterpret_cast<const int4*>(c->d_mc_blk + 4 * ntiles);
    prof_begin(c, ST_MC_EMIT);
    launch_tiles<EmitK>(c->mc_tile, ntiles, c->stream, c->g, (const unsigned*)c->d_mc_bits,
                        (const unsigned char*)c->d_mc_cls, nr, wp, ntiles, agg, sup, c->d_mc_tot, c->d_mc_nodes, (int)c->cap_mc_nodes, c->d_mc_word, c->h_mc_tot);
    c->launches++;
    cudaError_t e = cudaGetLastError();
    prof_end(c, ST_MC_EMIT);
    if (e != cudaSuccess) return e;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    prof_begin(c, ST_MC_TRIS);
    launch_pdl(k_mc_tris, (sms > 0 ? sms : kSms) * c->mc_tris_per_sm, 256, 0, c->stream, c->g, c->d_A, c->d_levelf, c->d_mc_nodes,
               (const int*)c->d_mc_tot, (int)c->cap_mc_nodes, (int)c->cap_tris, (const int2*)c->d_mc_word, wp,
               c->d_tris, c->d_verts, c->d_vnrm, (int)c->cap_verts);
    c->launches++;
    e = cudaGetLastError();
    prof_end(c, ST_MC_TRIS);
    return e;
}

cudaError_t launch_mesh_copy(ftr_ctx* c, float* verts, float* nrm, int32_t* tris) {
    if (!verts && !nrm && !tris) return cudaSuccess;
    const int64_t words = 3 * (c->n_verts > c->n_tris ? c->n_verts : c->n_tris);
    const int64_t blocks = (words / 4 + 255) / 256;
    k_mesh_copy<<<(unsigned)(blocks < 1 ? 1 : (blocks > kSms * 8 ? kSms * 8 : blocks)), 256, 0, c->stream>>>(
        c->d_verts, c->d_vnrm, c->d_tris, c->n_verts, c->n_tris, verts, nrm, tris);
    c->launches++;
    return cudaGetLastError();
}

cudaError_t launch_raise_flag(ftr_ctx* c, int* flag) {
    k_raise_flag<<<1, 1, 0, c->stream>>>(flag);
    c->launches++;
    return cudaGetLastError();
}

cudaError_t launch_mc_classes(ftr_ctx* c, uint8_t* out_dev) {
    const int64_t ncell = (int64_t)(c->g.n[0] - 1) * (c->g.n[1] - 1) * (c->g.n[2] - 1);
    k_mc_classes<<<(unsigned)((ncell + 255) / 256), 256, 0, c->stream>>>(c->g, c->d_A, c->d_levelf, out_dev);
    c->launches++;
    return cudaGetLastError();
}

}  // namespace ftr

// Register/shared-memory building blocks of the batched 1D FFT passes.
//
// The 3D transforms of Sec. III-B (forward FFT of the three components of V,
// inverse FFT of the filtered spectrum) are done as one pass per axis.  Every
// pass moves tiles of F independent length-N lines through one CTA:
//
//   N = N1 * N2,  n = N2 n1 + j,  k = k1 + N1 k2
//   X[k1 + N1 k2] = sum_j W_N^{j k1} W_N2^{j k2} sum_n1 x[N2 n1 + j] W_N1^{n1 k1}
//
// step 1: thread j of a line holds x[N2 n1 + j] (n1 < N1) in registers, does
//         a length-N1 DFT, multiplies by W_N^{j k1} and parks the values in
//         shared memory;
// step 2: thread k1 of a line gathers the N2 values for its k1 and does a
//         length-N2 DFT, ending with X[k1 + N1 k2] (k2 < N2) in registers.
// The small DFTs are unrolled Cooley-Tukey compositions of radix-2/3/4
// butterflies whose twiddles are compile-time indices into a 96-entry table
// (every small length used divides 96).  Forward transforms use
// exp(-2 pi i nk/N); inverse ones exp(+2 pi i nk/N) without scaling.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <set>
#include <utility>

#include "ftr_internal.h"

namespace ftr {

// W_96^j = exp(-2 pi i j / 96), a constant table of each translation unit,
// copied once per device by the unit's init function from the table the
// device computed in float64 (launch_twiddle, n = 96).
static __constant__ float2 c_w96[96];

static inline cudaError_t upload_w96_table(const float2* w96_dev) {
    return cudaMemcpyToSymbol(c_w96, w96_dev, 96 * sizeof(float2), 0, cudaMemcpyDeviceToDevice);
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// i * a
__device__ __forceinline__ float2 cmuli(float2 a) { return make_float2(-a.y, a.x); }

// Multiply by W_R^m (SIGN = -1 forward, +1 inverse) with m, R compile-time
// after unrolling.
template <int R, int SIGN>
__device__ __forceinline__ float2 tw_small(float2 v, int m) {
    const int j = ((m % R) * (96 / R)) % 96;
    if (j == 0) return v;
    if (j == 48) return make_float2(-v.x, -v.y);
    if (j == 24) return SIGN < 0 ? make_float2(v.y, -v.x) : make_float2(-v.y, v.x);   // -i / +i
    if (j == 72) return SIGN < 0 ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);   // +i / -i
    float2 w = c_w96[j];
    if (SIGN > 0) w.y = -w.y;
    return cmul(v, w);
}

template <int R, int SIGN>
struct Dft;

template <int SIGN>
struct Dft<1, SIGN> {
    __device__ __forceinline__ static void run(float2 (&)[1]) {}
};

template <int SIGN>
struct Dft<2, SIGN> {
    __device__ __forceinline__ static void run(float2 (&x)[2]) {
        float2 a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    }
};

template <int SIGN>
struct Dft<3, SIGN> {
    __device__ __forceinline__ static void run(float2 (&x)[3]) {
        // W_3 = -1/2 + SIGN i sqrt(3)/2
        const float s3 = 0.866025403784438647f * (float)SIGN;
        float2 a = x[0], b = x[1], c = x[2];
        float2 t1 = cadd(b, c);
        float2 t2 = make_float2(a.x - 0.5f * t1.x, a.y - 0.5f * t1.y);
        float2 d = csub(b, c);
        float2 t3 = make_float2(-d.y * s3, d.x * s3);   // i * SIGN * sqrt(3)/2 * (b - c)
        x[0] = cadd(a, t1);
        x[1] = cadd(t2, t3);
        x[2] = csub(t2, t3);
    }
};

template <int SIGN>
struct Dft<4, SIGN> {
    __device__ __forceinline__ static void run(float2 (&x)[4]) {
        float2 a = x[0], b = x[1], c = x[2], d = x[3];
        float2 s0 = cadd(a, c), s1 = csub(a, c);
        float2 s2 = cadd(b, d), s3 = csub(b, d);
        float2 r = cmuli(s3);                 // i (b - d)
        if (SIGN < 0) r = make_float2(-r.x, -r.y);
        x[0] = cadd(s0, s2);
        x[2] = csub(s0, s2);
        x[1] = cadd(s1, r);                   // (a - c) + SIGN i (b - d)
        x[3] = csub(s1, r);
    }
};

template <int R>
struct FirstFactor {
    static constexpr int value = (R % 4 == 0) ? 4 : ((R % 2 == 0) ? 2 : 3);
};

// Composite length: R = P Q, n = Q n1 + n2, k = k1 + P k2.
template <int R, int SIGN>
struct Dft {
    static constexpr int P = FirstFactor<R>::value;
    static constexpr int Q = R / P;
    __device__ __forceinline__ static void run(float2 (&x)[R]) {
        float2 y[R];
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            float2 t[P];
#pragma unroll
            for (int n1 = 0; n1 < P; ++n1) t[n1] = x[Q * n1 + n2];
            Dft<P, SIGN>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < P; ++k1) y[n2 * P + k1] = tw_small<R, SIGN>(t[k1], n2 * k1);
        }
#pragma unroll
        for (int k1 = 0; k1 < P; ++k1) {
            float2 u[Q];
#pragma unroll
            for (int n2 = 0; n2 < Q; ++n2) u[n2] = y[n2 * P + k1];
            Dft<Q, SIGN>::run(u);
#pragma unroll
            for (int k2 = 0; k2 < Q; ++k2) x[k1 + P * k2] = u[k2];
        }
    }
};

// Split of each supported line length into N1 (step-1 DFT) x N2 (step-2 DFT).
template <int N> struct Plan;
template <> struct Plan<32>  { static constexpr int N1 = 4,  N2 = 8; };
template <> struct Plan<48>  { static constexpr int N1 = 6,  N2 = 8; };
template <> struct Plan<64>  { static constexpr int N1 = 8,  N2 = 8; };
template <> struct Plan<96>  { static constexpr int N1 = 12, N2 = 8; };
template <> struct Plan<128> { static constexpr int N1 = 16, N2 = 8; };
template <> struct Plan<192> { static constexpr int N1 = 12, N2 = 16; };
template <> struct Plan<256> { static constexpr int N1 = 16, N2 = 16; };
template <> struct Plan<384> { static constexpr int N1 = 24, N2 = 16; };
template <> struct Plan<512> { static constexpr int N1 = 32, N2 = 16; };

__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Minimum resident CTAs per SM requested from the register allocator for the
// 16-line passes: what 80 registers per thread allow while the transform still
// fits in them (a spill of a few values at 384 points): three (24 warps) up to
// 256, two (24 warps) at 384, where the y and z pass otherwise take 121-145
// registers and run 12 warps (156 + 204 us, with the budget 119 + 171); one above.
template <int N>
struct MinCtas {
    static constexpr int value = N <= 256 ? 3 : (N <= 384 ? 2 : 1);
};
// The same register budget per thread for other tile heights F (lines per
// CTA): F = 8 asks for twice the CTAs of F = 16, F = 32 half (at least one).
template <int N, int F>
struct MinCtasF {
    static constexpr int raw = MinCtas<N>::value * 16 / F;
    static constexpr int value = raw < 1 ? 1 : raw;
};

// Raise a kernel's dynamic shared-memory limit to `bytes`, once per device.
template <class K>
inline cudaError_t ensure_smem(K kernel, size_t bytes, int device) {
    static std::mutex mu;
    static std::set<std::pair<const void*, int>> done;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair((const void*)kernel, device);
    if (done.count(key)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.insert(key);
    return e;
}

__host__ __device__ constexpr int make_odd(int v) { return (v & 1) ? v : v + 1; }

// Shared-memory exchange layout for F lines of length N: element (f, j, k1)
// at f + P1 k1 + P2 j.  P1 and P2 are odd so that 16 consecutive lanes that
// vary any one of f, j or k1 touch 16 different 8-byte bank pairs.  EIGHT: 16 lanes
// of step 1 are 8 lines x 2 values of j instead (the inverse x pass), and P2 is 8
// modulo 16 for them.
template <int N, int F, bool EIGHT = false>
struct Xchg {
    static constexpr int N1 = Plan<N>::N1, N2 = Plan<N>::N2;
    static constexpr int NT = cmax(N1, N2);               // threads per line
    static constexpr int P1 = make_odd(F + 1);
    static constexpr int P2 = EIGHT ? (P1 * N1 + 7) / 16 * 16 + 8 : make_odd(P1 * N1);   // forward layout (j < N2, k1 < N1)
    static constexpr int P2R = make_odd(P1 * N2);         // swapped layout (j < N1, k1 < N2)
    static constexpr int SIZE = cmax(P2 * N2, P2R * N1);  // float2 elements
    __device__ __forceinline__ static int idx(int f, int j, int k1) { return f + P1 * k1 + P2 * j; }
    __device__ __forceinline__ static int idxr(int f, int j, int k1) { return f + P1 * k1 + P2R * j; }
};

// The threads of step 1 (and of step 2 in swapped roles) are the CTA's first F N2,
// thread t working on line t / N2 (or t % F), so that the others are whole warps:
// cut into lines of NT like step 2's, a third to a half of every warp's lanes idled
// where N1 > N2.  384^3: x 87 -> 75, y 119 -> 109, z 171 -> 152 us.  (Step 2 where N1 <
// N2 keeps lines of NT: packed lines of N1 = 12 were no faster, 18.3 -> 19.1 us for the
// inverse x pass of 192^3.)
//
// Step 1 of a length-N transform: regs hold x[N2 n1 + j]; afterwards the
// twiddled step-1 results sit in the exchange buffer.  tw = the axis table
// (W_N^m, then W_N^(j k1) as [k1 < N1][j < N2], then as [k1 < N2][j < N1]).
template <int N, int F, int SIGN, bool EIGHT = false>
__device__ __forceinline__ void fft_step1(float2 (&v)[Plan<N>::N1], int f, int j, float2* xs,
                                          const float2* __restrict__ tw) {
    using X = Xchg<N, F, EIGHT>;
    Dft<X::N1, SIGN>::run(v);
#pragma unroll
    for (int k1 = 0; k1 < X::N1; ++k1) {
        if (k1 == 0) {
            xs[X::idx(f, j, 0)] = v[0];
            continue;
        }
        float2 w = __ldg(&tw[N + k1 * X::N2 + j]);      // W^0 = 1 - 0 i for j = 0
        if (SIGN > 0) w.y = -w.y;
        xs[X::idx(f, j, k1)] = cmul(v[k1], w);
    }
}

// Step 2: thread i (< N1) of line f gathers its column and ends with
// X[i + N1 k2] in out[k2].
template <int N, int F, int SIGN, bool EIGHT = false>
__device__ __forceinline__ void fft_step2(float2 (&out)[Plan<N>::N2], int f, int i, const float2* xs) {
    using X = Xchg<N, F, EIGHT>;
#pragma unroll
    for (int j = 0; j < X::N2; ++j) out[j] = xs[X::idx(f, j, i)];
    Dft<X::N2, SIGN>::run(out);
}

// Swapped-role steps (N = N2 * N1) used to run a second transform straight
// from the registers that step 2 left: thread i holds x[i + N1 n1'] (n1' < N2).
template <int N, int F, int SIGN>
__device__ __forceinline__ void fft_step1_swapped(float2 (&v)[Plan<N>::N2], int f, int j, float2* xs,
                                                  const float2* __restrict__ tw) {
    using X = Xchg<N, F>;
    Dft<X::N2, SIGN>::run(v);
#pragma unroll
    for (int k1 = 0; k1 < X::N2; ++k1) {
        if (k1 == 0) {
            xs[X::idxr(f, j, 0)] = v[0];
            continue;
        }
        float2 w = __ldg(&tw[2 * N + k1 * X::N1 + j]);
        if (SIGN > 0) w.y = -w.y;
        xs[X::idxr(f, j, k1)] = cmul(v[k1], w);
    }
}

template <int N, int F, int SIGN>
__device__ __forceinline__ void fft_step2_swapped(float2 (&out)[Plan<N>::N1], int f, int i, const float2* xs) {
    using X = Xchg<N, F>;
#pragma unroll
    for (int j = 0; j < X::N1; ++j) out[j] = xs[X::idxr(f, j, i)];
    Dft<X::N1, SIGN>::run(out);
}

// z-planes [zl, zh) that can hold non-zero data after the splat: the slab of
// touched bricks (meta[2] .. meta[3]) widened to multiples of 16 planes, the
// tile height of the y and z passes.  Empty when no brick was touched.
__device__ __forceinline__ void live_z_range(const int* __restrict__ meta, int& zl, int& zh) {
    const int bmin = meta[2], bmax = meta[3];
    if (bmax < 0) {
        zl = zh = 0;
        return;
    }
    zl = (bmin * 8) & ~15;
    zh = ((bmax + 1) * 8 + 15) & ~15;
}

// Which 16-row groups of z-plane z hold non-zero V: bit y / 16 (meta[kMetaRows +
// z / 8], set by the splat per touched brick).  Rows outside them transform to
// zero along x: the x pass neither computes nor writes their spectra and the y
// pass takes zeros in their place.  A body in its box touches about 45 % of the
// (y, z) rows inside its live slab.
__device__ __forceinline__ unsigned live_rows(const int* __restrict__ meta, int z) {
    return (unsigned)meta[kMetaRows + (z >> 3)];
}

// Ask L2 to fetch the 128-byte line holding p (no register is written, so
// later loads of the line find it in L2 instead of DRAM).
__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// A pass may ask for the input of the CTA `ahead` places later in launch order (about
// the one that takes this CTA's place) to be brought to L2, so that its loads wait for
// L2 and not for DRAM: inverse x of 384^3 117 -> 108 us; split precision (bf16x3) z 307
// -> 270, inverse x 173 -> 163.  Not where a half spectrum of `elems` fits L2 and mostly
// is there (256^3: split-precision z 87 -> 90), nor in the other passes (float32 z of
// 384^3 152 -> 162, y passes no gain).  Block index, or x = -1: none.
__device__ __forceinline__ int2 later_block(int ahead, int64_t elems) {
    if (elems * (int64_t)sizeof(float2) <= (int64_t)128 << 20) return make_int2(-1, -1);
    const int id = (int)(blockIdx.x + gridDim.x * blockIdx.y) + ahead;
    if (id >= (int)(gridDim.x * gridDim.y)) return make_int2(-1, -1);
    return make_int2(id % (int)gridDim.x, id / (int)gridDim.x);
}

// Element of the inverse x passes' staged half spectra, [k_x][16 rows]: the halves of
// odd k_x are exchanged, so that 16 lanes of 8 rows x 2 consecutive k_x touch 16
// different bank pairs.  With EIGHT above: half of the pass's shared-memory wavefronts
// were conflicts; 256^3 32.7 -> 30.7 us, 384^3 110 -> 99 (bf16x3 157 -> 146).
__device__ __forceinline__ int staged_at(int kx, int row) { return 16 * kx + (row ^ ((kx & 1) << 3)); }

// L2 eviction priorities for the passes' intermediates: a pass reads its
// input once (evict first: the lines are dead after) and writes the next
// pass's input (evict last: kept in L2 in preference, so that more of it is
// still there when the next pass reads it).
__device__ __forceinline__ uint64_t l2_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ float2 ld_l2hint(const float2* a, uint64_t pol) {
    float2 v;
    asm volatile("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ void st_l2hint(float2* a, float2 v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(a), "f"(v.x), "f"(v.y), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void st_l2hint(float* a, float v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(pol) : "memory");
}

// Signed frequency index of bin k on an axis of length n (Nyquist -> -n/2).
__device__ __forceinline__ int signed_bin(int k, int n) { return k < n / 2 ? k : k - n; }

}  // namespace ftr

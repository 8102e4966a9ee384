// Position of a point in node units, shared by the point ingest and the
// allocation-free level: t = (X - b_min) / h - 1/2 per axis, its floor, its
// fraction and the acceptance test, with every decision equal to that of the
// float64 quotient.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace ftr {

// t = (X - b_min) / h - 1/2 per axis.  The float64 product with 1/h is exact
// enough for the stencil offsets; wherever it could round to the other side
// of a decision (the acceptance bounds, floor(t), floor(t + 1/2)) the
// quotient is recomputed with a true division, so every decision equals that
// of (X - b_min) / h in float64.
__device__ __forceinline__ double node_t(double x, double bmin, double h, double inv_h, double n) {
    double t = (x - bmin) * inv_h - 0.5;
    const double band = 1e-9 * (1.0 + fabs(t));
    const double fr = t - floor(t);
    const double fh = (t + 0.5) - floor(t + 0.5);
    if (fr < band || fr > 1.0 - band || fh < band || fh > 1.0 - band || fabs(t - 1.0) < band ||
        fabs(t - (n - 2.0)) < band)
        t = (x - bmin) / h - 0.5;
    return t;
}

// The same t without float64 arithmetic: x - b_min exactly as a sum of two
// floats (two-sum), times 1/h held as a float pair, gives t = th + tl with an
// error below 1e-11 for t < 2^9 (|tl| stays below ~6e-5).  The fraction
// r = (th - floor th) + tl is rounded once, by at most 2^-25 as the float64 one
// would be: where t lies past the node that th falls short of, r is formed from
// the exact difference to that node (1 + 5e-5 would round by 2^-24), and below
// floor th the small remainder is the only other rounding.  floor(t), the
// nearest-node round-up and acceptance (floor(t) in [1, n - 3]) follow from it.
// Returns false when r lies within 1e-6 of 0, 1/2 or 1, where node_t decides
// instead.
__device__ __forceinline__ bool node_t_pair(float x, float bmin, float ih, float ih_lo, int& fl, float& fr,
                                            bool& up) {
    const float s = x - bmin;
    const float bb = s - x;
    const float e = (x - (s - bb)) + (-bmin - bb);
    const float p = s * ih;
    const float tl = fmaf(s, ih, -p) + fmaf(s, ih_lo, e * ih);
    const float th = p - 0.5f;
    if (!(fabsf(th) < 8388608.0f)) return false;   // NaN, inf or huge: float64 path
    const float f = floorf(th);
    float r = (th - f) + tl;                       // th - f is exact
    int fi = (int)f;
    const float band = 1e-6f;
    if (fabsf(r) < band || fabsf(r - 1.0f) < band || fabsf(r - 0.5f) < band) return false;
    if (r < 0.f) {
        r += 1.0f;
        fi -= 1;
    } else if (r > 1.0f) {
        r = (th - f - 1.0f) + tl;                  // th - f - 1 is exact too
        fi += 1;
    }
    fl = fi;
    fr = r;
    up = r > 0.5f;
    return true;
}

}  // namespace ftr

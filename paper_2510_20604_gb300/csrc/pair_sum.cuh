// Sums held as pairs of floats s + c: products are exact (FMA), additions carry
// their rounding error (Knuth's two-sum) in c, about 48 bits altogether.  FP64 runs at 2 FMA per
// cycle and SM on this GPU, so long FP32 dot products are summed this way and
// only their few partial sums are FP64.
#pragma once

#include <algorithm>
#include <cmath>

#include "rwc_common.cuh"

namespace rwc {

// Norm that an inner solve gives its residual: a power of two (no bit of a result
// depends on it) near the root of the mean degree.  The sums' terms are r r and
// r r / d, and at the end of a solve r r is 1e-16 for 10^6 vertices, so with |r|
// = 1 the rounding errors that a pair carries leave FP32's range at degrees of
// 1e15 and the terms themselves at 1e28.  Within 2^-20 .. 2^50, so that r r stays
// in range too.
inline double inner_scale(const DevGraph &g) {
    const int e = (int)std::lround(0.5 * std::log2(g.vol / (double)g.n));
    return std::ldexp(1.0, std::max(-20, std::min(50, e)));
}

struct Pair { float s, c; };
__device__ __forceinline__ void pair_add(Pair &a, float p, float low) {
    const float t = __fadd_rn(a.s, p);
    const float z = __fsub_rn(t, a.s);
    const float err = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, z)), __fsub_rn(p, z));
    a.c = __fadd_rn(a.c, __fadd_rn(err, low));
    a.s = t;
}
// a += x y
__device__ __forceinline__ void pair_fma(Pair &a, float x, float y) {
    const float p = __fmul_rn(x, y);
    pair_add(a, p, __fmaf_rn(x, y, -p));
}

}  // namespace rwc

// Sums held as pairs of floats s + c: products are exact (FMA), additions carry
// their rounding error in c, about 48 bits altogether.  FP64 runs at 2 FMA per
// cycle and SM on this GPU, so long FP32 dot products are summed this way and
// only their few partial sums are FP64.
#pragma once

namespace rwc {

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

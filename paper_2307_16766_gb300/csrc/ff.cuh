// ff.cuh -- float-float arithmetic: unevaluated sums hi + lo of two floats,
// built from the error-free transformations TwoSum (Knuth) and TwoProduct
// (by FMA): about 48 significant bits at FP32 issue cost (one FP64 warp
// instruction takes 64 cycles on each SM sub-partition of GB300, an FP32 one
// a single cycle).  The band kernel forms the wave amplitudes and the
// right-hand side with FP32 and FP16 storage in them: their projections
// S dU/dn cancel (an acoustic wave has a small entropy part), and plain FP32
// lost accuracy there.
#pragma once
#include "collide.cuh"

namespace lbmgb {

struct FF {
    float h, l;
};
__device__ __forceinline__ FF ff_fast(float a, float b)      // |a| >= |b|
{
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ FF ff_two_sum(float a, float b)
{
    const float s = a + b, z = s - a;
    return {s, (a - (s - z)) + (b - z)};
}
__device__ __forceinline__ FF ff_prod(float a, float b)
{
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ FF ff_add(FF x, FF y)
{
    const FF s = ff_two_sum(x.h, y.h), t = ff_two_sum(x.l, y.l);
    const FF u = ff_fast(s.h, s.l + t.h);
    return ff_fast(u.h, u.l + t.l);
}
__device__ __forceinline__ FF ff_neg(FF x) { return {-x.h, -x.l}; }
__device__ __forceinline__ FF ff_mul(FF x, float b)
{
    const FF p = ff_prod(x.h, b);
    return ff_fast(p.h, fmaf(x.l, b, p.l));
}
__device__ __forceinline__ FF ff_mul(FF x, FF y)
{
    const FF p = ff_prod(x.h, y.h);
    return ff_fast(p.h, fmaf(x.h, y.l, fmaf(x.l, y.h, p.l)));
}
__device__ __forceinline__ double ff_to_double(FF x) { return double(x.h) + double(x.l); }
__device__ __forceinline__ FF ff_const(const float (&c)[2]) { return {c[0], c[1]}; }
__device__ __forceinline__ FF ff_scale(FF x, float p2) { return {x.h * p2, x.l * p2}; }   // p2: a power of 2
__device__ __forceinline__ FF ff_split(double d)
{
    const float h = float(d);
    return {h, float(d - double(h))};
}

__device__ __forceinline__ FF ff_sub(FF x, FF y) { return ff_add(x, ff_neg(y)); }

}  // namespace lbmgb

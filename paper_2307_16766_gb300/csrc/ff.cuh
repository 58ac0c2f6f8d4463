// ff.cuh -- float-float arithmetic: unevaluated sums hi + lo of two floats,
// built from the error-free transformations TwoSum (Knuth) and TwoProduct
// (by FMA): about 48 significant bits at FP32 issue cost (one FP64 warp
// instruction takes 64 cycles on each SM sub-partition of GB300, an FP32 one
// a single cycle).  The band kernel forms the wave amplitudes and the
// right-hand side with FP32 and FP16 storage in them: their projections
// S dU/dn cancel (an acoustic wave has a small entropy part), and plain FP32
// lost accuracy there.  The macroscopic fields of FP32 and FP16 populations
// are summed in them too (macros_ff).
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
// The double a float stands for, by its bits (a conversion instruction goes
// through the FP64 pipe); denormals, infinities and NaN are converted.
__device__ __forceinline__ double float_widen(float x)
{
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    if (m - 1u < 0x007fffffu || m >= 0x7f800000u) return double(x);
    return __hiloint2double(int((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), int(m << 29));
}
__device__ __forceinline__ double ff_widen(FF x) { return float_widen(x.h) + float_widen(x.l); }
__device__ __forceinline__ double ff_pack(FF x)
{
    return __hiloint2double(__float_as_int(x.h), __float_as_int(x.l));
}
__device__ __forceinline__ FF ff_unpack(double v)
{
    return {__int_as_float(__double2hiint(v)), __int_as_float(__double2loint(v))};
}
__device__ __forceinline__ FF ff_const(const float (&c)[2]) { return {c[0], c[1]}; }
__device__ __forceinline__ FF ff_scale(FF x, float p2) { return {x.h * p2, x.l * p2}; }   // p2: a power of 2
__device__ __forceinline__ FF ff_split(double d)
{
    const float h = float(d);
    return {h, float(d - double(h))};
}

__device__ __forceinline__ FF ff_sub(FF x, FF y) { return ff_add(x, ff_neg(y)); }
// x + y with the low parts added plainly: for sums whose terms do not all
// cancel (error ~2^-47 of the larger term)
__device__ __forceinline__ FF ff_acc(FF x, FF y)
{
    const FF s = ff_two_sum(x.h, y.h);
    return {s.h, s.l + (x.l + y.l)};
}
__device__ __forceinline__ FF ff_norm(FF x) { return ff_two_sum(x.h, x.l); }
// 1 / x: the float reciprocal and one Newton step
__device__ __forceinline__ FF ff_rcp(FF x)
{
    const float r = 1.0f / x.h;
    const float e = fmaf(-x.l, r, fmaf(-x.h, r, 1.0f));
    return ff_fast(r, r * e);
}

// Macroscopic fields (Eq. macro) of FP32 / FP16 populations in float-float:
// h are the stored values (FP16: g / w), U = (drho, u_x, u_y, theta - 1).
// Opposite pairs first (their sums and differences are exact in
// float-float), then per class (even parts) and per speed (odd parts), so
// that a node takes 54 accumulations instead of 140; the weights of scaled
// storage and the lattice constants enter as float-float constants.
template <int LAT, typename S>
__device__ __forceinline__ void macros_ff(const Geom& G, const float* h, double* U)
{
    using L = Lat<LAT>;
    constexpr bool SC = Store<S>::SCALED;
    constexpr int NC = L::NCLS;
    auto konst = [](double v) -> FF { return {float(v), float(v - double(float(v)))}; };
    // sums with a flag "still empty" (resolved when the loop is unrolled)
    struct Sum {
        FF v{0.0f, 0.0f};
        bool any = false;
        __device__ void add(FF x)
        {
            v = any ? ff_acc(v, x) : x;
            any = true;
        }
    };
    Sum E[NC], X[SC ? NC : 4], Y[SC ? NC : 4];
    E[0].add(FF{h[0], 0.0f});
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const int k = L::cls(i), cx = L::cx(i), cy = L::cy(i);
        const FF e = ff_two_sum(h[i], h[i + 1]), o = ff_two_sum(h[i], -h[i + 1]);
        E[k].add(e);
        // scaled storage: odd sums per class, the factor |c_x| (a power of 2
        // or 3) taken in; otherwise per |c_x| and |c_y|
        if (cx) {
            const FF s = cx > 0 ? o : ff_neg(o);
            const int a = cx > 0 ? cx : -cx;
            if (SC) X[k].add(a == 1 ? s : a == 2 ? ff_scale(s, 2.0f) : ff_acc(ff_scale(s, 2.0f), s));
            else X[a].add(s);
        }
        if (cy) {
            const FF s = cy > 0 ? o : ff_neg(o);
            const int a = cy > 0 ? cy : -cy;
            if (SC) Y[k].add(a == 1 ? s : a == 2 ? ff_scale(s, 2.0f) : ff_acc(ff_scale(s, 2.0f), s));
            else Y[a].add(s);
        }
    }
    FF s0, sx, sy, se{0.0f, 0.0f};
    if constexpr (SC) {
        s0 = ff_mul(ff_norm(E[0].v), konst(L::wcls(0)));
        sx = sy = FF{0.0f, 0.0f};
#pragma unroll
        for (int k = 1; k < NC; ++k) {
            const FF w = konst(L::wcls(k)), e = ff_mul(ff_norm(E[k].v), w);
            s0 = ff_acc(s0, e);
            if (L::THERMAL) se = ff_acc(se, ff_mul(e, float(L::c2cls(k))));
            sx = ff_acc(sx, ff_mul(ff_norm(X[k].v), w));
            sy = ff_acc(sy, ff_mul(ff_norm(Y[k].v), w));
        }
    } else {
        s0 = E[0].v;
#pragma unroll
        for (int k = 1; k < NC; ++k) {
            const FF e = ff_norm(E[k].v);
            s0 = ff_acc(s0, e);
            if (L::THERMAL) se = ff_acc(se, ff_mul(e, float(L::c2cls(k))));
        }
        const FF x3 = ff_norm(X[3].v), y3 = ff_norm(Y[3].v);
        sx = ff_acc(ff_acc(X[1].v, ff_scale(X[2].v, 2.0f)), ff_acc(ff_scale(x3, 2.0f), x3));
        sy = ff_acc(ff_acc(Y[1].v, ff_scale(Y[2].v, 2.0f)), ff_acc(ff_scale(y3, 2.0f), y3));
    }
    s0 = ff_norm(s0);
    sx = ff_norm(sx);
    sy = ff_norm(sy);
    const FF rho = ff_add(ff_split(G.rho0), s0), ir = ff_rcp(rho);
    const FF Ux{G.ref ? G.uref_f[0] : 0.0f, 0.0f}, Uy{G.ref ? G.uref_f[1] : 0.0f, 0.0f};
    if (G.ref) {                        // as moments_of_sums
        sx = ff_sub(sx, ff_mul(s0, Ux.h));
        sy = ff_sub(sy, ff_mul(s0, Uy.h));
    }
    const FF vx = ff_mul(sx, ir), vy = ff_mul(sy, ir);
    U[0] = ff_widen(s0);
    U[1] = ff_widen(vx);
    U[2] = ff_widen(vy);
    if (G.ref) {
        U[1] += double(Ux.h);
        U[2] += double(Uy.h);
    }
    U[3] = 0.0;
    if (L::THERMAL) {
        se = ff_norm(se);
        // rho |v|^2 (+ 2 rho U.v) = (sx + 2 rho U_x) v_x + ...
        FF qx = sx, qy = sy;
        FF e = ff_sub(se, ff_mul(s0, konst(2.0 * L::CS2)));
        if (G.ref) {
            qx = ff_add(sx, ff_scale(ff_mul(rho, Ux.h), 2.0f));
            qy = ff_add(sy, ff_scale(ff_mul(rho, Uy.h), 2.0f));
            e = ff_sub(e, ff_mul(s0, ff_add(ff_prod(Ux.h, Ux.h), ff_prod(Uy.h, Uy.h))));
        }
        e = ff_sub(e, ff_add(ff_mul(qx, vx), ff_mul(qy, vy)));
        U[3] = ff_widen(ff_mul(ff_mul(e, ir), konst(0.5 / L::CS2)));
    }
}

}  // namespace lbmgb

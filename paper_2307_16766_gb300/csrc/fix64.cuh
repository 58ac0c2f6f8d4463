// fix64.cuh -- FP64 sums and the FP64 collision on the integer pipe.
//
// One FP64 warp instruction takes 64 cycles of an SM sub-partition on GB300,
// an integer one 1 to 2, so the FP64 update (467 FP64 instructions a D2Q37
// node) was bound by that pipe at a tenth of the memory bandwidth.  Here the
// additions and the products with the velocities' small integer components
// are done in block fixed point: the numbers of one node are written as
// integers times a common power of two taken from the largest of them, added
// exactly, and rounded once when they become doubles again.  FP64 is left for
// what is a product of two fields: the macros, the monomial coefficients of
// the equilibrium and two operations per stored population (142 instructions a
// D2Q37 node: 140 of the 174 us of an update of 1024x512, the rest waits on it).
//
// D2Q37 1024x512, 20 steps with initial fields and read-out: 10.43 -> 3.96 ms
// (the bulk update 461 -> 174 us).  Errors of the velocities against extended
// precision (80 bits), geometric mean over 8 to 16 flows of 20 to 80 steps,
// tau 0.55 to 1.1, beside those of FP64 sums and an FP64 equilibrium:
//   a stream, periodic   D2Q9 1.1e-17, 1.4e-17; D2Q17 1.2e-17, 3.8e-17; D2Q37 9.1e-18, 1.1e-16
//   ... through CBC sides D2Q9 1.3e-17, 2.0e-17; D2Q17 1.1e-17, 2.6e-17; D2Q37 9.3e-18, 3.8e-17
//   from rest            D2Q9 1.7e-19, 2.4e-19; D2Q17 9.5e-20, 2.4e-19; D2Q37 3.4e-20, 3.2e-19
// (u_x; u_y, density and temperature are no further off in any row either).
#pragma once
#include "lbm_internal.cuh"

namespace lbmgb {

// Biased exponent of a double from its high word.
__device__ __forceinline__ int fx_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Block exponents the fixed-point forms take: no infinities, NaN or overflow
// above, no denormal results below; everything else goes to the FP64 forms.
__device__ __forceinline__ bool fx_range(int e) { return e >= 128 && e <= 1900; }

// The leading bit of a number of the block's largest exponent.  kFxTop: the
// base of the units of the non-equilibrium moments (up to 259 populations in
// one value, counted with their factors) and of the equilibrium, which follow
// the size of the values (fx_block, fx_equilibrium).
// fx_top: the sums of populations.  With 56 of them the operands' rounding was
// of the size of the stored populations' own (D2Q37: velocities of a decaying
// pulse 20 % further off than with FP64 sums).  D2Q9 and D2Q17 have room for 57
// in 64 bits (at most 20 populations in one sum, counted with c); D2Q37 (52)
// takes 58 and adds its per-speed sums (at most 14 each) in 128 bits.
// kFxFloat: the sums of FP32 populations (52 of them in 64 bits).
constexpr int kFxTop = 54, kFxFloat = 56;
template <int LAT>
constexpr int fx_top() { return Lat<LAT>::Q > 17 ? 58 : 57; }

// v in units of 2^(emax - 1023 - T), rounded to nearest (truncation is a
// drift that adds up over the steps); |v| < 2^(emax - 1022), emax >= 128.
template <int T>
__device__ __forceinline__ long long fx_of(double v, int emax)
{
    const int hi = __double2hiint(v);
    const unsigned long long m =
        ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << (T - 51);
    const int d = emax - ((hi >> 20) & 0x7ff);
    const long long a = (long long)(((m >> (d < 63 ? d : 63)) + 1) >> 1), s = hi >> 31;
    return (a ^ s) - s;
}

// A float in the same units, rounded down (the sums of a read-out feed nothing
// back): exact if its last bit is above the unit.  Denormals count as zero
// (fx_block_float).
template <int T>
__device__ __forceinline__ long long fx_of(float v, int emax)
{
    const int b = __float_as_int(v), s = b >> 31, e = (b >> 23) & 0xff;
    const int m = e ? (((b & 0x7fffff) | 0x800000) ^ s) - s : 0;
    const int d = emax - (1023 - 127) + (62 - T) - e;
    return (long long)((unsigned long long)(unsigned)m << 39) >> (d < 63 ? d : 63);
}

// The same for T = kFxTop with 32 more bits below, truncated; |v| < 2^(emax - 1014).
__device__ __forceinline__ __int128 fx_wide_of(double v, int emax)
{
    const int hi = __double2hiint(v);
    const unsigned long long m =
        (unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v);
    // m << (32 + kFxTop - 52 - d) as high and low words, eight places higher first
    constexpr int UP = 32 + kFxTop - 52 + 8;
    const int d = emax - ((hi >> 20) & 0x7ff) + 8, n = d < 95 ? d : 95;
    unsigned long long h = m >> (64 - UP), l = m << UP;
    if (n >= 64) {
        l = h >> (n - 64);
        h = 0;
    } else if (n > 0) {
        l = l >> n | h << (64 - n);
        h >>= n;
    }
    const __int128 a = (__int128)((unsigned __int128)h << 64 | l);
    return hi < 0 ? -a : a;
}

// c_s^2, its square and its inverse in units of 2^-60: of the double that the
// moments are formed with, on D2Q9 (isothermal: no moment takes it) of 1/3.
template <int LAT>
struct FxCs2 {
    long long c, cc, inv;
    constexpr FxCs2() : c(0), cc(0), inv(0)
    {
        if (!Lat<LAT>::THERMAL) {
            c = ((1LL << 60) + 1) / 3;
            inv = 3LL << 60;
            return;
        }
        double v = Lat<LAT>::CS2;
        int e = 0;
        for (; v < 4503599627370496.0; ++e) v *= 2.0;      // c_s^2 = m 2^-e, 2^52 <= m < 2^53
        const __int128 m = (__int128)v;
        c = (long long)((m << 60) >> e);
        cc = (long long)((m * m) >> (2 * e - 60));
        inv = (long long)((((__int128)1 << (60 + e)) + m / 2) / m);
    }
};

// x k 2^-60, |x| < 2^95
__device__ __forceinline__ __int128 fx_mul(__int128 x, long long k)
{
    return ((__int128)(long long)(x >> 32) * k >> 28) + ((__int128)(unsigned)x * k >> 60);
}

// x units of 2^(emax - 1023 - T) as a double, rounded to nearest.
template <int T>
__device__ __forceinline__ double fx_double(long long x, int emax)
{
    const long long s = x >> 63;
    unsigned long long a = (unsigned long long)((x ^ s) - s);
    const int n = __clzll((long long)a);
    a <<= (n & 63);
    const unsigned long long m = (a >> 11) + ((a >> 10) & 1);       // 53 bits, the leading one included
    const unsigned e = (unsigned)(emax + (63 - T) - 1 - n) << 20;
    const unsigned h = (unsigned)(m >> 32) + e + ((unsigned)s & 0x80000000u);
    return a ? __hiloint2double((int)h, (int)(unsigned)m) : 0.0;
}

// The same for a sum that may be beyond 63 bits, which drops 8 of them then.
template <int T>
__device__ __forceinline__ double fx_double(__int128 x, int emax)
{
    const bool big = (long long)(x >> 64) != (long long)x >> 63;
    return fx_double<T>(big ? (long long)((x + 128) >> 8) : (long long)x, big ? emax + 8 : emax);
}

// A positive double as a 53-bit integer times a power of two, m 2^e, and the
// weights of a lattice's classes as such.
struct FxConst {
    long long m;
    int e;
};
template <int LAT>
struct FxWeights {
    FxConst w[Lat<LAT>::NCLS];
    constexpr FxWeights() : w()
    {
        for (int k = 0; k < Lat<LAT>::NCLS; ++k) {
            double v = Lat<LAT>::wcls(k);
            int e = 0;
            for (; v < 4503599627370496.0; --e) v *= 2.0;      // 2^52
            w[k].m = (long long)v;
            w[k].e = e;
        }
    }
};

// w times x units of 2^(emax - 1023 - kFxTop) as a double: 64 leading bits of
// the product, rounded to nearest.
__device__ __forceinline__ double fx_scaled(long long x, FxConst w, int emax)
{
    const long long s = x >> 63;
    unsigned long long a = (unsigned long long)((x ^ s) - s);
    const int n = __clzll((long long)a);
    a = __umul64hi(a << (n & 63), (unsigned long long)w.m << 11);       // in [2^62, 2^64)
    const int k = a >> 63 ? 0 : 1;
    a <<= k;
    const unsigned long long m = (a >> 11) + ((a >> 10) & 1);           // 53 bits, the leading one included
    const unsigned e = (unsigned)(emax + w.e + (116 - kFxTop) - 1 - n - k) << 20;
    const unsigned h = (unsigned)(m >> 32) + e + ((unsigned)s & 0x80000000u);
    return x ? __hiloint2double((int)h, (int)(unsigned)m) : 0.0;
}

// The block exponent of populations get(0..Q-1), or 0 if the fixed-point
// forms do not take them.  Populations that are all zero count as any block.
template <int LAT, typename Get>
__device__ __forceinline__ int fx_block(Get&& get)
{
    int emax = 0;
    unsigned any = 0;
#pragma unroll
    for (int i = 0; i < Lat<LAT>::Q; ++i) {
        const double v = get(i);
        const int hi = __double2hiint(v) & 0x7fffffff;
        emax = hi > emax ? hi : emax;
        any |= unsigned(hi) | unsigned(__double2loint(v));
    }
    emax >>= 20;
    return any == 0 ? 1023 : fx_range(emax) ? emax : 0;
}

// The same, and in `up` how many bits further down than kFxTop the sums of
// fx_neq_sums may go: per class the largest weight a moment's sum gives it in
// all, with the class's own exponent, stays below 2^63 then (2^-20 of the
// block's binade a unit of the bound; 54 + up between 53 and 61).
template <int LAT, typename Get>
__device__ __forceinline__ int fx_block(Get&& get, int& up)
{
    using L = Lat<LAT>;
    int top[L::NCLS];
    unsigned any = 0;
#pragma unroll
    for (int k = 0; k < L::NCLS; ++k) top[k] = 0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const double v = get(i);
        const int hi = __double2hiint(v) & 0x7fffffff;
        top[L::cls(i)] = max(top[L::cls(i)], hi);
        any |= unsigned(hi) | unsigned(__double2loint(v));
    }
    int emax = 0;
#pragma unroll
    for (int k = 0; k < L::NCLS; ++k) {
        top[k] >>= 20;
        emax = max(emax, top[k]);
    }
    // sum over a class of |c_x c_y|, |c_x^2 - c_y^2|, |c_x^2|, |(|c|^2 - 5) c_x|, |(|c|^2 - 4 c_s^2) c_x|
    constexpr int W37[8] = {0, 8, 12, 16, 27, 42, 38, 116}, W17[5] = {0, 8, 12, 52, 45}, W9[3] = {0, 2, 4};
    int bound = 16;
#pragma unroll
    for (int k = 1; k < L::NCLS; ++k)
        bound += ((L::Q == 37 ? W37[k % 8] : L::Q == 17 ? W17[k % 5] : W9[k % 3]) << 20) >> min(emax - top[k], 31);
    up = min(__clz(bound) - 4, 7);
    return any == 0 ? 1023 : fx_range(emax) ? emax : 0;
}

// The same of FP32 populations: 0 only for infinities and NaN.  A block below
// 2^-67 (the front of a pulse) is lifted by 2^lift first, so that denormals
// count in it; in the others they are below the unit.
template <int LAT>
__device__ __forceinline__ int fx_block_float(float* g, int& lift)
{
    int emax = 0;
    lift = 0;
#pragma unroll
    for (int i = 0; i < Lat<LAT>::Q; ++i) emax = max(emax, __float_as_int(g[i]) & 0x7fffffff);
    if (emax == 0) return 1023;
    if (emax < 60 << 23) {
        lift = 96;
#pragma unroll
        for (int i = 0; i < Lat<LAT>::Q; ++i) g[i] *= 7.9228162514264338e28f;
        emax = __float_as_int(__int_as_float(emax) * 7.9228162514264338e28f);
    }
    const int e = emax >> 23;
    return e < 255 ? e + (1023 - 127) : 0;
}

// The sums of Eq. macro: s0 = sum g, (sx, sy) = sum g c, se = sum g |c|^2, of
// populations lifted by 2^lift.
template <int LAT, int T = fx_top<LAT>(), typename Get>
__device__ __forceinline__ void fx_sums(Get&& get, int emax, double& s0, double& sx, double& sy, double& se,
                                        int lift = 0)
{
    using L = Lat<LAT>;
    long long E[L::NCLS], X[4] = {0, 0, 0, 0}, Y[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < L::NCLS; ++k) E[k] = 0;
    E[0] = fx_of<T>(get(0), emax);
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const int cx = L::cx(i), cy = L::cy(i);
        const long long p = fx_of<T>(get(i), emax), m = fx_of<T>(get(i + 1), emax), o = p - m;
        E[L::cls(i)] += p + m;
        if (cx > 0) X[cx] += o;
        if (cx < 0) X[-cx] -= o;
        if (cy > 0) Y[cy] += o;
        if (cy < 0) Y[-cy] -= o;
    }
    using A = std::conditional_t<(T > 57), __int128, long long>;
    A a0 = 0;
    __int128 ae = 0;
#pragma unroll
    for (int k = 0; k < L::NCLS; ++k) {
        a0 += E[k];
        if (L::THERMAL) ae += (__int128)L::c2cls(k) * E[k];
    }
    emax -= lift;
    s0 = fx_double<T>(a0, emax);
    sx = fx_double<T>(X[1] + A(2) * X[2] + A(3) * X[3], emax);
    sy = fx_double<T>(Y[1] + A(2) * Y[2] + A(3) * Y[3], emax);
    se = L::THERMAL ? fx_double<T>(ae, emax) : 0.0;
}

// x 2^-88 as a double.
__device__ __forceinline__ double fx_double_scaled(__int128 x)
{
    const long long h = (long long)(x >> 64);
    const int n = 65 - __clzll(h ^ (h >> 63));      // one place more than the high word's bits, and
    const bool wide = h != (long long)x >> 63;      // none if the low word holds the number
    return fx_double<88>(wide ? (long long)(x >> n) : (long long)x, wide ? 1023 + n : 1023);
}

// The same sums of FP16 storage, h = g / w (FP16 values in float); false if
// one is not finite.  An FP16 value is an integer of 41 bits times 2^-24: two
// floats, hi 2^-4 + lo 2^-24, whose sums over a class (16 counted with c) are
// exact in FP32; then the classes' weights in units of 2^-64 (a double's last
// bit or 2^-65) on 32-bit parts, and one rounding each.
template <int LAT>
__device__ __forceinline__ bool fx_sums_scaled(const float* h, double& s0, double& sx, double& sy, double& se)
{
    using L = Lat<LAT>;
    constexpr int N = L::NCLS;
    float E[N][2], X[N][2], Y[N][2];
#pragma unroll
    for (int k = 0; k < N; ++k) E[k][0] = E[k][1] = X[k][0] = X[k][1] = Y[k][0] = Y[k][1] = 0.0f;
    auto split = [](float v, float* p) {
        p[0] = fmaf(v, 16.0f, 12582912.0f) - 12582912.0f;       // to an integer (1.5 2^23)
        p[1] = fmaf(p[0], -1048576.0f, v * 16777216.0f);
    };
    split(h[0], E[0]);
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const int k = L::cls(i);
        const float cx = float(L::cx(i)), cy = float(L::cy(i));
        float p[2], m[2];
        split(h[i], p);
        split(h[i + 1], m);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            E[k][q] += p[q] + m[q];
            if (L::cx(i)) X[k][q] = fmaf(cx, p[q] - m[q], X[k][q]);
            if (L::cy(i)) Y[k][q] = fmaf(cy, p[q] - m[q], Y[k][q]);
        }
    }
    // (hi 2^20 + lo) (wh 2^32 + wl): four sums of 32-bit products each
    struct Sum {
        long long a = 0, b = 0, c = 0, d = 0;
        __device__ void add(int hi, int lo, long long w)
        {
            const int wl = int(unsigned(w)), wh = int((w - wl) >> 32);
            a += (long long)hi * wh;
            b += (long long)hi * wl;
            c += (long long)lo * wh;
            d += (long long)lo * wl;
        }
        __device__ double get() const
        {
            return fx_double_scaled((((__int128)a << 20) + c << 32) + ((__int128)b << 20) + d);
        }
    } S, SX, SY, SE;
    float all = 0.0f;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const long long w = (long long)(L::wcls(k) * 18446744073709551616.0);     // below 1/2
        all += E[k][1];
        const int hi = __float2int_rn(E[k][0]), lo = __float2int_rn(E[k][1]);
        S.add(hi, lo, w);
        if (k == 0) continue;
        if (L::THERMAL) SE.add(hi, lo, L::c2cls(k) * w);
        SX.add(__float2int_rn(X[k][0]), __float2int_rn(X[k][1]), w);
        SY.add(__float2int_rn(Y[k][0]), __float2int_rn(Y[k][1]), w);
    }
    s0 = S.get();
    sx = SX.get();
    sy = SY.get();
    se = L::THERMAL ? SE.get() : 0.0;
    return isfinite(all);               // an infinity leaves NaN in lo
}

// Moments (Eq. macro) of populations get(i); false if they are out of range.
template <int LAT, typename Get>
__device__ __forceinline__ bool fx_moments(Get&& get, double rho0, int ref, double Ux, double Uy,
                                           Moments<LAT, double>& m)
{
    const int emax = fx_block<LAT>(get);
    if (emax == 0) return false;
    double s0, sx, sy, se;
    fx_sums<LAT>(get, emax, s0, sx, sy, se);
    m = moments_of_sums<LAT, double>(s0, sx, sy, se, rho0, ref, Ux, Uy);
    return true;
}

// The equilibrium (see eq_poly) of moments m held against w rho0, in the
// monomials of (c_x, c_y):
//   g^eq_i / w_i = sum over a + b <= ORDER of m_ab c_x^a c_y^b,
// one value at a time to put(i, w, x, e): g^eq_i = fx_scaled(x, w, e).  False,
// with nothing put, if the coefficients are out of the fixed-point range.
// (jx, jy), se: rho u and sum g |c|^2.  All velocities share the coefficients'
// rounding, which in a uniform stream adds up over the steps; so the ones that
// carry mass, momentum and energy are not formed in FP64 but closed in the
// integers, with q = 3 m_40 + 3 m_04 + m_22:
//   m_20 + m_02 = (se - 2 c_s^2 s) / (2 c_s^4) - 2 c_s^2 q  (thermal lattices),
//   m_00 = s - c_s^2 (m_20 + m_02) - c_s^4 q,
//   m_10 = j_x / c_s^2 - c_s^2 (3 m_30 + m_12),  m_01 likewise,
// which is what the expansion's coefficients are, so that g^eq carries s, j
// and se whatever the rounding of the others, of 1 / c_s^2, u and theta.
template <int LAT, typename Put>
__device__ __forceinline__ bool fx_equilibrium(const Moments<LAT, double>& m, double jx, double jy, double se, Put&& put)
{
    using L = Lat<LAT>;
    using W = __int128;
    constexpr bool O3 = L::ORDER >= 3, O4 = L::ORDER >= 4;
    constexpr double ics2 = 1.0 / L::CS2;
    const double X = m.ux * ics2, Y = m.uy * ics2;
    const EqPoly<double> e = eq_poly<LAT, double>(m.ux * X + m.uy * Y, m.dT);
    // coefficients: with p = c_x X + c_y Y and q = |c|^2,
    // s0 + rho [A0 + B0' q + C0' q^2 + (A2 + B2' q) p^2 + p^4 / 24] and
    // rho [(A1 + B1' q) p + p^3 / 6]
    constexpr int NM = O4 ? 15 : O3 ? 10 : 6;
    double c[NM];
    const double rX = jx * ics2, rY = jy * ics2, XX = X * X, XY = X * Y, YY = Y * Y;
    const double rA2 = m.rho * e.A2, rB0 = m.rho * (e.B0 * ics2);
    c[0] = m.s0;                            // 1, without the closing part
    c[1] = rX;                              // x (its size; the value is closed)
    c[2] = rY;                              // y
    c[3] = rB0 + rA2 * XX;                  // x^2
    c[4] = rB0 + rA2 * YY;                  // y^2
    c[5] = 2.0 * rA2 * XY;                  // x y
    if constexpr (O3) {
        const double B1 = e.B1 * ics2;
        c[6] = rX * (B1 + (1.0 / 6.0) * XX);    // x^3
        c[7] = rY * (B1 + (1.0 / 6.0) * YY);    // y^3
        c[8] = rY * (B1 + 0.5 * XX);            // x^2 y
        c[9] = rX * (B1 + 0.5 * YY);            // x y^2
    }
    if constexpr (O4) {
        const double rB2 = m.rho * (e.B2 * ics2), rC0 = m.rho * (e.C0 * (ics2 * ics2)), r4 = m.rho * (1.0 / 24.0);
        c[10] = rC0 + XX * (rB2 + r4 * XX);                                     // x^4
        c[11] = rC0 + YY * (rB2 + r4 * YY);                                     // y^4
        c[12] = 2.0 * rC0 + (rB2 * (XX + YY) + (6.0 * r4) * (XX * YY));         // x^2 y^2
        c[13] = XY * (2.0 * rB2 + (4.0 * r4) * XX);                             // x^3 y
        c[14] = XY * (2.0 * rB2 + (4.0 * r4) * YY);                             // x y^3
    }
    int ec = 0;
#pragma unroll
    for (int k = 0; k < NM; ++k) ec = max(ec, fx_exp(c[k]));
    if (L::THERMAL) ec = max(ec, fx_exp(se));
    if (ec == 0) ec = 1023;                 // all zero
    if (!fx_range(ec)) return false;
    // the largest value that can arise, in units of 2^(ec - 1022 - 20): the
    // factors are the monomials' at the outermost velocities, with the closing
    // parts' shares (c_s^2 < 0.7).  The unit is chosen so that it stays below
    // 2^63 (seven to minus one bits below that of ec and kFxTop).
    constexpr int F[15] = {1, 3, 3, 10, 10, 4, 34, 34, 12, 12, 83, 83, 17, 27, 27};
    int bound = 16;
#pragma unroll
    for (int k = 0; k < NM; ++k) bound += (F[k] << 20) >> min(ec - fx_exp(c[k]), 31);
    if (L::THERMAL) bound += (1 << 20) >> min(ec - fx_exp(se), 31);
    ec -= __clz(bound) - 4;
    constexpr FxCs2<LAT> K{};
    W v[NM];
#pragma unroll
    for (int k = 3; k < NM; ++k) v[k] = fx_wide_of(c[k], ec);
    const W s = fx_wide_of(c[0], ec);
    W q = 0, tr = v[3] + v[4];
    if constexpr (O4) q = 3 * (v[10] + v[11]) + v[12];
    if constexpr (L::THERMAL) {
        const W d = v[3] - v[4];
        tr = (fx_mul(fx_mul(fx_wide_of(se, ec) - 2 * fx_mul(s, K.c), K.inv), K.inv) >> 1) - 2 * fx_mul(q, K.c);
        v[3] = (tr + d) >> 1;
        v[4] = (tr - d) >> 1;
    }
    v[0] = s - fx_mul(tr, K.c);
    v[1] = fx_mul(fx_wide_of(jx, ec), K.inv);
    v[2] = fx_mul(fx_wide_of(jy, ec), K.inv);
    if constexpr (O3) {
        v[1] -= fx_mul(3 * v[6] + v[9], K.c);
        v[2] -= fx_mul(3 * v[7] + v[8], K.c);
    }
    if constexpr (O4) v[0] -= fx_mul(q, K.cc);
    // the parts below are rounded to 64 bits by adding this and dropping 32
    const W half = W(1) << 31;
    v[0] += half;
    // per axis: even x^2 + x^4 and odd x + x^3 parts at |c| = 0 .. 3
    W fx[4], fy[4], gx[4], gy[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        fx[a] = W(a * a) * v[3];
        fy[a] = W(a * a) * v[4];
        gx[a] = W(a) * v[1] + (a ? half : 0);
        gy[a] = W(a) * v[2] + (a ? half : 0);
        if constexpr (O3) {
            gx[a] += W(a * a * a) * v[6];
            gy[a] += W(a * a * a) * v[7];
        }
        if constexpr (O4) {
            fx[a] += W(a * a * a * a) * v[10];
            fy[a] += W(a * a * a * a) * v[11];
        }
    }
    constexpr FxWeights<LAT> wt{};
    put(0, wt.w[0], (long long)(v[0] >> 32), ec);
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const int cx = L::cx(i), cy = L::cy(i), a = cx < 0 ? -cx : cx, b = cy < 0 ? -cy : cy;
        W Ev = (v[0] + fx[a]) + fy[b], Ox = gx[a], Oy = gy[b], Xy = 0;
        if (a && b) {
            Xy = W(a * b) * v[5] + half;
            if constexpr (O3) {
                Ox += W(a * b * b) * v[9];
                Oy += W(a * a * b) * v[8];
            }
            if constexpr (O4) {
                Ev += W(a * a * b * b) * v[12];
                Xy += W(a * a * a * b) * v[13] + W(a * b * b * b) * v[14];
            }
        }
        const long long ev = (long long)(Ev >> 32), xy = (long long)(Xy >> 32), ox = (long long)(Ox >> 32),
                        oy = (long long)(Oy >> 32);
        const long long E = cx * cy < 0 ? ev - xy : ev + xy;
        const long long O = (cx < 0 ? -ox : ox) + (cy < 0 ? -oy : oy);
        put(i, wt.w[L::cls(i)], E + O, ec);
        put(i + 1, wt.w[L::cls(i)], E - O, ec);
    }
    return true;
}

// BGK collision (Eq. bgk) of the populations get(i) of a node with moments m;
// post-collision values go to put(i, value).  g^eq is rounded before g is taken
// from it, so that a node at equilibrium stays there: with the residue of an
// unrounded product, omega > 1 moves it by a unit in the last place each step.
template <int LAT, typename Get, typename Put>
__device__ __forceinline__ bool fx_relax(const Moments<LAT, double>& m, double om, Get&& get, Put&& put)
{
    return fx_equilibrium<LAT>(m, m.sx, m.sy, m.se, [&](int i, FxConst w, long long x, int e) {
        const double g = get(i);
        put(i, fma(om, fx_scaled(x, w, e) - g, g));
    });
}

// neq_moments (collide.cuh) with its sums in fixed point; get(i) in range.
// The third moments are sum g (|c|^2 - 5) c + (5 - 4 c_s^2) sum g c, the product
// with the constant in 128 bits: the two parts all but cancel.  The operands go
// `up` bits below kFxTop (fx_block; usually three to five).  Without them p_xy
// was up to 3.5 times, q up to 3.5 times on D2Q17, as far off as the sums over
// g - g^eq in FP64.
template <int LAT, typename Get>
__device__ __forceinline__ void fx_neq_sums(Get&& get, int emax, int up, double& pxy, double& dxy, double& pxx,
                                            double& pyy, double& rx, double& ry)
{
    using L = Lat<LAT>;
    constexpr int T = 61;                       // the finest unit
    emax -= up;
    auto of = [&](double v) { return fx_of<T>(v, emax + (T - kFxTop)); };
    long long axy = 0, ad = 0, axx = 0, ayy = 0, ax = 0, ay = 0, jx = 0, jy = 0;
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const int cx = L::cx(i), cy = L::cy(i), c2 = cx * cx + cy * cy;
        const long long p = of(get(i)), m = of(get(i + 1)), e = p + m, o = p - m;
        axy += (long long)(cx * cy) * e;
        if (L::THERMAL) {
            ad += (long long)(cx * cx - cy * cy) * e;
            ax += (long long)((c2 - 5) * cx) * o;
            ay += (long long)((c2 - 5) * cy) * o;
            jx += (long long)cx * o;
            jy += (long long)cy * o;
        } else {
            axx += (long long)(cx * cx) * e;
            ayy += (long long)(cy * cy) * e;
        }
    }
    pxy = fx_double<kFxTop>(axy, emax);
    if (L::THERMAL) {
        dxy = fx_double<kFxTop>(ad, emax);
        // the constant in units of 2^-60 (below 2^62); the product's part alone
        // may leave 64 bits, the sum does not
        constexpr FxCs2<LAT> C{};
        constexpr long long K = (5LL << 60) - 4 * C.c;
        const __int128 half = (__int128)1 << 59;
        auto third = [&](long long a, long long j) {
            return (long long)((unsigned long long)a + (unsigned long long)(((__int128)j * K + half) >> 60));
        };
        rx = fx_double<kFxTop>(third(ax, jx), emax);
        ry = fx_double<kFxTop>(third(ay, jy), emax);
        pxx = pyy = 0.0;
    } else {
        pxx = fx_double<kFxTop>(axx, emax);
        pyy = fx_double<kFxTop>(ayy, emax);
        dxy = rx = ry = 0.0;
    }
}

}  // namespace lbmgb

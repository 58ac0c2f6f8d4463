// collide.cuh -- the per-node update shared by the bulk kernels (bulk.cu)
// and the band kernel (boundary.cu): plain pull, moments, BGK collision.
#pragma once
#include "dual.cuh"
#include "lbm_internal.cuh"

namespace lbmgb {

// 1/tau and rho0 in the precision of arithmetic type C (float-based types
// take the float-rounded values).
template <typename C>
__device__ __forceinline__ C omega_of(const Geom& G)
{
    if constexpr (sizeof(typename DualTraits<C>::Value) == 4) return C(G.omega_f);
    else return C(G.omega);
}
template <typename C>
__device__ __forceinline__ C rho0_of(const Geom& G)
{
    if constexpr (sizeof(typename DualTraits<C>::Value) == 4) return C(G.rho0_f);
    else return C(G.rho0);
}

// The reference velocity of the stored populations in the precision of C.
template <typename C>
__device__ __forceinline__ C uref_of(const Geom& G, int k)
{
    if constexpr (sizeof(typename DualTraits<C>::Value) == 4) return C(G.uref_f[k]);
    else return C(G.uref[k]);
}

// The reference velocity the populations of storage S are held against, as
// a double: the value in the storage's arithmetic (float-rounded for FP32
// and FP16), so that every kernel shifts by the same equilibrium.
template <typename S>
__host__ __device__ __forceinline__ double stored_ref(const Geom& G, int k)
{
    if constexpr (sizeof(typename Store<S>::C) == 4) return double(G.uref_f[k]);
    else return G.uref[k];
}

// Moments of the stored populations g of a node (the grid's reference; REF =
// false compiles the plain shift only, for kernels instantiated per form).
template <int LAT, typename C, bool REF = true>
__device__ __forceinline__ Moments<LAT, C> moments_G(const Geom& G, const C* g)
{
    return moments<LAT, C>(g, rho0_of<C>(G), REF ? G.ref : 0, uref_of<C>(G, 0), uref_of<C>(G, 1));
}

// Viscous stress sigma' = -(1 - 1/(2 tau)) sum c c (f - f^eq) (Eq. LaplaceU)
// and heat flux q = (1 - 1/(2 tau)) 1/2 sum (f - f^eq) |c-u|^2 (c-u)
// (Eqs. heatflux, LaplaceT; the equilibrium part of the central third
// moment vanishes on the thermal lattices).
// FP64: the equilibria reproduce the Maxwellian moments through third order
// (second on D2Q9), so their share is taken in closed form,
//   sum f^eq c_a c_b = rho (u_a u_b + c_s^2 theta delta_ab),
//   sum f^eq |c|^2 c_a = rho u_a (|u|^2 + 4 c_s^2 theta),
// instead of from 37 evaluated populations (500 more operations a node, 30 us
// of FP64 issue in a band tile).  f - f^eq carries no mass, momentum or
// energy: on the thermal lattices its stress is traceless, formed from
// c_x^2 - c_y^2 with the large isotropic part cancelling pair by pair, and its
// third moment is that of (|c|^2 - 4 c_s^2) c, so that the rounding of rho, u
// and theta does not enter at their size.  With a reference the closed forms
// are differences from the reference's.
// FP32 and derivative numbers (EVAL) keep the sums over g - g^eq: the closed
// form is faster where the band kernel is all there is (256^2: 2.12 ms a pass,
// 2.20 with the sums) and slower beside a large bulk (1024x512: 3.48, 3.34; 96
// runs: 30.5, 29.8), and the gradients of short runs feel its different
// rounding.  FP16 storage and populations relative to a reference, where
// there are no gradients, take the closed form: 1024x512 with a reference 3.87 ms
// a pass (4.00 with the sums); FP16, 60 steps: 512x512 with an outlet 1.43 ms
// (1.53), 1024x512 with four sides 1.92 (2.03), 1600x1200 4.84 (4.91), 2048^2
// 9.06 (9.08).
template <int LAT, typename C, typename T>
__device__ __forceinline__ void neq_evaluated(const C* g, const Moments<LAT, C>& m, T fac, T* N)
{
    using L = Lat<LAT>;
    Moments<LAT, C> me = m;
    if constexpr (std::is_same_v<C, float>)
        // kept apart from the moments' and the collision's arithmetic, so that
        // every kernel contracts this one alike (a run of a batch repeats bit
        // for bit alone)
        asm volatile("" : "+f"(me.s0), "+f"(me.rho), "+f"(me.ux), "+f"(me.uy), "+f"(me.dT));
    C geq[L::Q];
    equilibrium<LAT, C>(me, geq);
    C pxx = 0, pxy = 0, pyy = 0, qx = 0, qy = 0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const C d = g[i] - geq[i];
        const C cx = C(L::cx(i)), cy = C(L::cy(i));
        pxx += cx * cx * d;
        pxy += cx * cy * d;
        pyy += cy * cy * d;
        if (L::THERMAL) {
            const C ex = cx - me.ux, ey = cy - me.uy;
            const C h = C(0.5) * d * (ex * ex + ey * ey);
            qx += h * ex;
            qy += h * ey;
        }
    }
    N[0] = -fac * T(pxx);
    N[1] = -fac * T(pxy);
    N[2] = -fac * T(pyy);
    N[3] = fac * T(qx);
    N[4] = fac * T(qy);
}

template <int LAT, typename C, typename T>
__device__ __forceinline__ void neq_close(const Moments<LAT, C>& m, T fac, T* N, C pxy, C dxy, C pxx, C pyy, C rx, C ry);

template <int LAT, typename C, typename T, bool EVAL = !std::is_same_v<C, double>>
__device__ __forceinline__ void neq_moments(const C* g, const Moments<LAT, C>& m, T fac, T* N)
{
    using L = Lat<LAT>;
    constexpr double cs2 = L::CS2;
    if constexpr (EVAL) return neq_evaluated<LAT, C, T>(g, m, fac, N);
    // sum g c_x c_y; sum g (c_x^2 - c_y^2) per class (thermal) or sum g c_a^2
    // (D2Q9); sum g (|c|^2 - 4 c_s^2) c_a
    C pxy = 0, dxy = 0, pxx = 0, pyy = 0, rx = 0, ry = 0;
#pragma unroll
    for (int k = 1; k < L::NCLS; ++k) {
        C d = 0;
#pragma unroll
        for (int i = 1; i < L::Q; i += 2) {
            if (L::cls(i) != k) continue;
            const int cx = L::cx(i), cy = L::cy(i), c2 = cx * cx + cy * cy;
            const C e = g[i] + g[i + 1];
            if (cx * cy) pxy += C(cx * cy) * e;
            if (!L::THERMAL) {
                if (cx) pxx += C(cx * cx) * e;
                if (cy) pyy += C(cy * cy) * e;
                continue;
            }
            if (cx * cx > cy * cy) d += e;
            if (cx * cx < cy * cy) d -= e;
            const C o = g[i] - g[i + 1];
            if (cx) rx += C((c2 - 4.0 * cs2) * cx) * o;
            if (cy) ry += C((c2 - 4.0 * cs2) * cy) * o;
        }
        // |c_x^2 - c_y^2| of the class
        const int c2 = L::c2cls(k), dd = c2 == 1 ? 1 : c2 == 4 ? 4 : c2 == 5 ? 3 : c2 == 9 ? 9 : c2 == 10 ? 8 : 0;
        if (L::THERMAL && dd) dxy += C(dd) * d;
    }
    neq_close<LAT, C, T>(m, fac, N, pxy, dxy, pxx, pyy, rx, ry);
}

// The closed-form equilibrium's share taken from the sums above.
template <int LAT, typename C, typename T>
__device__ __forceinline__ void neq_close(const Moments<LAT, C>& m, T fac, T* N, C pxy, C dxy, C pxx, C pyy, C rx, C ry)
{
    using L = Lat<LAT>;
    constexpr double cs2 = L::CS2;
    const C ux = m.ux, uy = m.uy;
    if (m.ref) {
        const C U2x = m.Ux * m.Ux, U2y = m.Uy * m.Uy, wx = m.vx * (ux + m.Ux), wy = m.vy * (uy + m.Uy);
        pxy -= m.s0 * (m.Ux * m.Uy) + m.rho * (m.Ux * m.vy + m.vx * uy);
        if (L::THERMAL) {
            const C rho0 = m.rho - m.s0, t4 = C(4.0 * cs2) * m.dT;
            const C W = ux * ux + uy * uy + t4, dW = wx + wy + t4;
            dxy -= m.s0 * (U2x - U2y) + m.rho * (wx - wy);
            rx -= (m.s0 * m.Ux + m.rho * m.vx) * W + rho0 * m.Ux * dW;
            ry -= (m.s0 * m.Uy + m.rho * m.vy) * W + rho0 * m.Uy * dW;
        } else {
            const C p = C(cs2) * m.s0;
            pxx -= p + m.s0 * U2x + m.rho * wx;
            pyy -= p + m.s0 * U2y + m.rho * wy;
        }
    } else {
        const C jx = m.rho * ux, jy = m.rho * uy;
        pxy -= jx * uy;
        if (L::THERMAL) {
            const C W = ux * ux + uy * uy + C(4.0 * cs2) * m.dT;
            dxy -= jx * ux - jy * uy;
            rx -= jx * W;
            ry -= jy * W;
        } else {
            const C p = C(cs2) * m.s0;
            pxx -= p + jx * ux;
            pyy -= p + jy * uy;
        }
    }
    if (L::THERMAL) {
        pxx = C(0.5) * dxy;
        pyy = -pxx;
    }
    N[0] = -fac * T(pxx);
    N[1] = -fac * T(pxy);
    N[2] = -fac * T(pyy);
    N[3] = N[4] = T(0);
    if (L::THERMAL) {
        N[3] = fac * T(C(0.5) * rx - (ux * pxx + uy * pxy));
        N[4] = fac * T(C(0.5) * ry - (ux * pxy + uy * pyy));
    }
}

// The elements at(0..Q-1) points to, as values.  FP16: the raw words of all of
// them first (the empty asm statements hold them), then the conversions; as
// one loop each load was waited for before the next (k_band with FP16 storage,
// D2Q37 512x512: 40 us a step, 23 us with the loads in flight together, FP32 21).
template <int LAT, typename S, typename C, bool LIVE, typename At>
__device__ __forceinline__ void load_all(At&& at, C* g)
{
    constexpr int Q = Lat<LAT>::Q;
    if constexpr (sizeof(S) == 2) {
        unsigned r[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const unsigned short* p = reinterpret_cast<const unsigned short*>(at(i));
            r[i] = LIVE ? *p : __ldg(p);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) asm volatile("" : "+r"(r[i]));
#pragma unroll
        for (int i = 0; i < Q; ++i) g[i] = C(Store<S>::value(__ushort_as_half((unsigned short)r[i])));
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if constexpr (LIVE) g[i] = C(Store<S>::value(*at(i)));
            else g[i] = C(Store<S>::load(at(i)));
        }
    }
}

// Plain pull of node (x, y) with periodic wrap-around of the sources.  LIVE:
// the previous step may still have been writing fin when this kernel started
// (early start), so the loads are ordinary ones, which the wait for that step
// orders; fin must not come from a const __restrict__ kernel parameter then,
// which would make them read-only loads again.
template <int LAT, typename S, typename C, bool LIVE = false>
__device__ __forceinline__ void pull_plain(const Geom& G, const Offsets& O, const S* fin, int x, int y, C* g)
{
    using L = Lat<LAT>;
    load_all<LAT, S, C, LIVE>(
        [&](int i) {
            int xs = x - L::cx(i), ys = y - L::cy(i);
            if (L::cx(i) && G.perx) xs = xs < 0 ? xs + G.nx : (xs >= G.nx ? xs - G.nx : xs);
            if (L::cy(i) && G.pery) ys = ys < 0 ? ys + G.ny : (ys >= G.ny ? ys - G.ny : ys);
            return fin + (O.st[i] + ys * G.nxp + xs);
        },
        g);
}

// The same with the plane offsets computed from the plane size (for kernels
// that serve several grids in one launch).
template <int LAT, typename S, typename C>
__device__ __forceinline__ void pull_plain_planes(const Geom& G, const S* __restrict__ fin, int x,
                                                  int y, C* g)
{
    using L = Lat<LAT>;
    const int plane = int(G.plane);
    load_all<LAT, S, C, false>(
        [&](int i) {
            int xs = x - L::cx(i), ys = y - L::cy(i);
            if (L::cx(i) && G.perx) xs = xs < 0 ? xs + G.nx : (xs >= G.nx ? xs - G.nx : xs);
            if (L::cy(i) && G.pery) ys = ys < 0 ? ys + G.ny : (ys >= G.ny ? ys - G.ny : ys);
            return fin + (L::plane_of(i) * plane + ys * G.nxp + xs);
        },
        g);
}

// Moments (Eq. macro) and BGK collision (Eq. bgk) of one node whose pulled
// populations are in g (already multiplied by w for scaled storage).  The
// post-collision value of velocity i goes to put(i, value); the moments of
// the pulled populations are returned.
// BGK collision of a node whose moments m are known; gi(i) gives the
// pre-collision population i (read as the pair loop needs it).
template <int LAT, typename C, typename Get, typename Put>
__device__ __forceinline__ void collide_given(const Geom& G, const Moments<LAT, C>& m, Get&& gi, Put&& put)
{
    using L = Lat<LAT>;
    constexpr int Q = L::Q;

    // BGK collide (Eq. bgk), one opposite pair at a time:
    // g^eq_{+-} = w (rho - rho0) + w rho (even +- odd) in p = c.u / c_s^2,
    // or, relative to a reference equilibrium (m.ref), w (Ev +- Od) of
    // eq_pair_ref.
    constexpr C ics2 = C(1.0 / L::CS2);
    constexpr C a3 = L::ORDER >= 3 ? C(1.0 / 6.0) : C(0);
    constexpr C a4 = L::ORDER >= 4 ? C(1.0 / 24.0) : C(0);
    const C uxs = m.ux * ics2, uys = m.uy * ics2;
    const EqPoly<C> e = eq_poly<LAT, C>(m.ux * uxs + m.uy * uys, m.dT);
    const C om = omega_of<C>(G);
    const bool ref = m.ref != 0;
    EqDelta<C> de;
    C rho0r = C(0), Uxs = C(0), Uys = C(0), vxs = C(0), vys = C(0);
    if (ref) {
        Uxs = m.Ux * ics2;
        Uys = m.Uy * ics2;
        vxs = m.vx * ics2;
        vys = m.vy * ics2;
        de = eq_delta<LAT, C>(m.Ux * Uxs + m.Uy * Uys, C(2) * (m.Ux * vxs + m.Uy * vys) + m.vx * vxs + m.vy * vys,
                              m.dT);
        rho0r = m.rho - m.s0;
    }
    // g^eq of the pair (i, i + 1) of class k
    auto pair = [&](int i, C& gp, C& gm) {
        const int k = L::cls(i);
        const C xi2 = C(L::c2cls(k)) * ics2;
        if (ref) {
            const C P = C(L::cx(i)) * Uxs + C(L::cy(i)) * Uys, q = C(L::cx(i)) * vxs + C(L::cy(i)) * vys;
            C Ev, Od;
            eq_pair_ref<LAT, C>(e, de, xi2, P, q, m.s0, rho0r, Ev, Od);
            gp = C(L::w(i)) * (Ev + Od);
            gm = C(L::w(i)) * (Ev - Od);
            return;
        }
        const C a0 = e.A0 + xi2 * (e.B0 + e.C0 * xi2);
        const C a1 = e.A1 + e.B1 * xi2;
        const C a2 = e.A2 + e.B2 * xi2;
        C p;
        if (L::cx(i) == 0) p = C(L::cy(i)) * uys;
        else if (L::cy(i) == 0) p = C(L::cx(i)) * uxs;
        else p = C(L::cx(i)) * uxs + C(L::cy(i)) * uys;
        const C p2 = p * p;
        const C ev = a0 + p2 * (a2 + p2 * a4);
        const C od = p * (a1 + p2 * a3);
        const C ws0 = C(L::w(i)) * m.s0, wr = C(L::w(i)) * m.rho;
        gp = ws0 + wr * (ev + od);
        gm = ws0 + wr * (ev - od);
    };
    if (sizeof(typename DualTraits<C>::Value) == 8) {
        {
            const C geq = ref ? C(L::w(0)) * (m.s0 * (C(1) + e.A0) + rho0r * de.A0)
                              : C(L::w(0)) * (m.s0 + m.rho * e.A0);
            { const C g_ = gi(0); put(0, g_ + om * (geq - g_)); }
        }
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            C gp, gm;
            pair(i, gp, gm);
            { const C g_ = gi(i); put(i, g_ + om * (gp - g_)); }
            { const C g_ = gi(i + 1); put(i + 1, g_ + om * (gm - g_)); }
        }
    } else {
        // FP32 arithmetic.  Float-rounded weights and c_s^2 miss the discrete
        // moment identities by ~1e-8, which would make each collision leak
        // mass, momentum and energy at that relative rate.  The equilibrium
        // is therefore closed on the conserved moments: the |c| = 1 pairs
        // take the momentum and energy remainders and the rest velocity the
        // mass remainder (corrections of float-rounding size).
        C M0 = 0, Mx = 0, My = 0, Me = 0;
#pragma unroll
        for (int i = 5; i < Q; i += 2) {
            const int k = L::cls(i);
            C gp, gm;
            pair(i, gp, gm);
            const C sum = gp + gm, dif = gp - gm;
            M0 += sum;
            if (L::cx(i)) Mx += C(L::cx(i)) * dif;
            if (L::cy(i)) My += C(L::cy(i)) * dif;
            if (L::THERMAL) Me += C(L::c2cls(k)) * sum;
            { const C g_ = gi(i); put(i, g_ + om * (gp - g_)); }
            { const C g_ = gi(i + 1); put(i + 1, g_ + om * (gm - g_)); }
        }
        // |c| = 1 class: (1,0) and (-1,0) are velocities 1, 2; (0,1), (0,-1) are 3, 4
        C ex, ey;
        if (ref) {
            C Ev, Od;
            eq_pair_ref<LAT, C>(e, de, ics2, Uxs, vxs, m.s0, rho0r, Ev, Od);
            ex = C(L::w(1)) * Ev;
            eq_pair_ref<LAT, C>(e, de, ics2, Uys, vys, m.s0, rho0r, Ev, Od);
            ey = C(L::w(1)) * Ev;
        } else {
            const C a0 = e.A0 + ics2 * (e.B0 + e.C0 * ics2);
            const C a2 = e.A2 + e.B2 * ics2;
            const C px2 = uxs * uxs, py2 = uys * uys;
            const C ws0 = C(L::w(1)) * m.s0, wr = C(L::w(1)) * m.rho;
            ex = ws0 + wr * (a0 + px2 * (a2 + px2 * a4));
            ey = ws0 + wr * (a0 + py2 * (a2 + py2 * a4));
        }
        if (L::THERMAL) {
            const C d = C(0.25) * (m.se - Me - C(2) * (ex + ey));
            ex += d;
            ey += d;
        }
        const C ox = C(0.5) * (m.sx - Mx), oy = C(0.5) * (m.sy - My);
        { const C g_ = gi(1); put(1, g_ + om * (ex + ox - g_)); }
        { const C g_ = gi(2); put(2, g_ + om * (ex - ox - g_)); }
        { const C g_ = gi(3); put(3, g_ + om * (ey + oy - g_)); }
        { const C g_ = gi(4); put(4, g_ + om * (ey - oy - g_)); }
        const C geq0 = m.s0 - M0 - C(2) * (ex + ey);
        { const C g_ = gi(0); put(0, g_ + om * (geq0 - g_)); }
    }

}

// The same collision for storage that holds h_i = g_i / w_i (FP16), done in
// those scaled variables so that no population is multiplied by w_i on the
// way in or divided by it on the way out: the moments are sums of w_i h_i
// (w_i c_i folded into one constant), and h^eq_i = g^eq_i / w_i =
// (rho - rho0) + rho (even +- odd) carries no weight.  FP32 arithmetic, with
// the conserved-moment closure of the FP32 path above (the closure sums take
// w_i back in).  put(i, value) receives h*_i.
template <int LAT, bool REF, typename Put>
__device__ __forceinline__ void collide_scaled(const Geom& G, const float* h, Put&& put)
{
    using L = Lat<LAT>;
    using C = float;
    constexpr int Q = L::Q;
    C s0 = 0, sx = 0, sy = 0, se = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        s0 += C(L::w(i)) * h[i];
        if (L::cx(i)) sx += C(L::w(i) * L::cx(i)) * h[i];
        if (L::cy(i)) sy += C(L::w(i) * L::cy(i)) * h[i];
        if (L::THERMAL && i) se += C(L::w(i) * (L::cx(i) * L::cx(i) + L::cy(i) * L::cy(i))) * h[i];
    }
    const Moments<LAT, C> m = moments_of_sums<LAT, C>(s0, sx, sy, se, rho0_of<C>(G), REF ? G.ref : 0,
                                                      uref_of<C>(G, 0), uref_of<C>(G, 1));
    constexpr C ics2 = C(1.0 / L::CS2);
    constexpr C a3 = L::ORDER >= 3 ? C(1.0 / 6.0) : C(0);
    constexpr C a4 = L::ORDER >= 4 ? C(1.0 / 24.0) : C(0);
    const C uxs = m.ux * ics2, uys = m.uy * ics2;
    const EqPoly<C> e = eq_poly<LAT, C>(m.ux * uxs + m.uy * uys, m.dT);
    const C om = omega_of<C>(G);
    const bool ref = m.ref != 0;
    EqDelta<C> de;
    C rho0r = C(0), Uxs = C(0), Uys = C(0), vxs = C(0), vys = C(0);
    if (ref) {
        Uxs = m.Ux * ics2;
        Uys = m.Uy * ics2;
        vxs = m.vx * ics2;
        vys = m.vy * ics2;
        de = eq_delta<LAT, C>(m.Ux * Uxs + m.Uy * Uys, C(2) * (m.Ux * vxs + m.Uy * vys) + m.vx * vxs + m.vy * vys,
                              m.dT);
        rho0r = m.rho - m.s0;
    }
    C M0 = 0, Mx = 0, My = 0, Me = 0;
#pragma unroll
    for (int i = 5; i < Q; i += 2) {
        const int k = L::cls(i);
        const C xi2 = C(L::c2cls(k)) * ics2;
        C hp, hm;
        if (ref) {
            const C P = C(L::cx(i)) * Uxs + C(L::cy(i)) * Uys, q = C(L::cx(i)) * vxs + C(L::cy(i)) * vys;
            C Ev, Od;
            eq_pair_ref<LAT, C>(e, de, xi2, P, q, m.s0, rho0r, Ev, Od);
            hp = Ev + Od;
            hm = Ev - Od;
        } else {
            const C a0 = e.A0 + xi2 * (e.B0 + e.C0 * xi2);
            const C a1 = e.A1 + e.B1 * xi2;
            const C a2 = e.A2 + e.B2 * xi2;
            C p;
            if (L::cx(i) == 0) p = C(L::cy(i)) * uys;
            else if (L::cy(i) == 0) p = C(L::cx(i)) * uxs;
            else p = C(L::cx(i)) * uxs + C(L::cy(i)) * uys;
            const C p2 = p * p;
            const C ev = a0 + p2 * (a2 + p2 * a4);
            const C od = p * (a1 + p2 * a3);
            hp = m.s0 + m.rho * (ev + od);
            hm = m.s0 + m.rho * (ev - od);
        }
        const C sum = hp + hm, dif = hp - hm;
        M0 += C(L::w(i)) * sum;
        if (L::cx(i)) Mx += C(L::w(i) * L::cx(i)) * dif;
        if (L::cy(i)) My += C(L::w(i) * L::cy(i)) * dif;
        if (L::THERMAL) Me += C(L::w(i) * L::c2cls(k)) * sum;
        put(i, h[i] + om * (hp - h[i]));
        put(i + 1, h[i + 1] + om * (hm - h[i + 1]));
    }
    // |c| = 1 class and the rest velocity close the conserved moments, in
    // unscaled units, then scaled
    C ex, ey;
    if (ref) {
        C Ev, Od;
        eq_pair_ref<LAT, C>(e, de, ics2, Uxs, vxs, m.s0, rho0r, Ev, Od);
        ex = C(L::w(1)) * Ev;
        eq_pair_ref<LAT, C>(e, de, ics2, Uys, vys, m.s0, rho0r, Ev, Od);
        ey = C(L::w(1)) * Ev;
    } else {
        const C a0 = e.A0 + ics2 * (e.B0 + e.C0 * ics2);
        const C a2 = e.A2 + e.B2 * ics2;
        const C px2 = uxs * uxs, py2 = uys * uys;
        const C ws0 = C(L::w(1)) * m.s0, wr = C(L::w(1)) * m.rho;
        ex = ws0 + wr * (a0 + px2 * (a2 + px2 * a4));
        ey = ws0 + wr * (a0 + py2 * (a2 + py2 * a4));
    }
    if (L::THERMAL) {
        const C d = C(0.25) * (m.se - Me - C(2) * (ex + ey));
        ex += d;
        ey += d;
    }
    const C ox = C(0.5) * (m.sx - Mx), oy = C(0.5) * (m.sy - My);
    constexpr C iw1 = C(1.0 / L::w(1));
    put(1, h[1] + om * ((ex + ox) * iw1 - h[1]));
    put(2, h[2] + om * ((ex - ox) * iw1 - h[2]));
    put(3, h[3] + om * ((ey + oy) * iw1 - h[3]));
    put(4, h[4] + om * ((ey - oy) * iw1 - h[4]));
    const C geq0 = m.s0 - M0 - C(2) * (ex + ey);
    put(0, h[0] + om * (geq0 * C(1.0 / L::w(0)) - h[0]));
}

template <int LAT, typename C, bool REF = false, typename Put>
__device__ __forceinline__ Moments<LAT, C> collide(const Geom& G, const C* g, Put&& put)
{
    const Moments<LAT, C> m = moments_G<LAT, C, REF>(G, g);
    collide_given<LAT, C>(G, m, [&](int i) -> const C& { return g[i]; }, put);
    return m;
}

}  // namespace lbmgb

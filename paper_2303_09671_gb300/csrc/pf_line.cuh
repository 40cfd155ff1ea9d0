// pf_line.cuh -- the explicit step on a strip of a 1D line held in one warp's
// registers (pf_batch.cu's batched fronts, pf_step1d.cu's single line).
//
// A warp holds 32 J consecutive cells, lane l the J cells l J .. l J + J - 1 as
// J/2 two-lane vectors: pair q is the cells (q, q + J/2), so that the right
// neighbour of pair q is pair q + 1 and only the last pair's right and the
// first pair's left neighbours come from another lane (one shuffle per value;
// no shared memory, no barrier).  The arithmetic is packed .f32x2 in FP32, and
// every face is evaluated once, by the cell to its left.  A step moves
// information by two cells, so after k steps the outermost 2k cells of the
// strip are stale: with J/2 steps between two exchanges exactly the first and
// the last lane are, and 30 of 32 lanes hold results.
//
// The method is that of pf_step.cu (Eq. phasefield_nonvar with the re-derived
// driving force at cells, the brackets of Eqs. cs_nonvar / cl_nonvar at faces,
// the conservative (c, d) update, forward Euler) in grid units: differences are
// not divided by dx, the stored rate is dx^2 dphi/dt and the fluxes are dx F.
#pragma once
#include <cfloat>
#include <cmath>
#include "pf_dual.cuh"
#include "pf_internal.cuh"
#include "pf_lanes.cuh"

namespace pf {

// ------------------------------------------------- two cells as one number
// A value of two cells: a two-lane vector V (float2, double2) or a value and a
// derivative of two cells, DV<V>.
template <typename V>
struct DV {
    V v, t;
};

// A lane of a Mono strip holds one FP64 cell per value instead of two: short FP64
// lines, whose cells are fewer than the lanes of the FP64 pipes.
struct Mono {};

template <typename E>
struct LineNum;   // element type -> vector types; M: the element in memory
template <>
struct LineNum<float> {
    using S = float;    // scalar without derivative
    using M = float;
    using V = float2;
    using X = float2;
    static constexpr int LANES = 2;
};
template <>
struct LineNum<Mono> {
    using S = double;
    using M = double;
    using V = double;
    using X = double;
    static constexpr int LANES = 1;
};
template <>
struct LineNum<double> {
    using S = double;
    using M = double;
    using V = double2;
    using X = double2;
    static constexpr int LANES = 2;
};
template <typename T>
struct LineNum<Dual<T>> {
    using S = T;
    using M = Dual<T>;
    using V = typename LineNum<T>::V;
    using X = DV<V>;
    static constexpr int LANES = 2;
};

#define PF_D __device__ __forceinline__
// one cell: its value is both "lanes", and a pair of values is its first
PF_D double x_lo(double a) { return a; }
PF_D double x_hi(double a) { return a; }
// (never contracted, so that every kernel that evaluates a cell gets the same bits)
PF_D double vadd(double a, double b) { return __dadd_rn(a, b); }
PF_D double vsub(double a, double b) { return __dsub_rn(a, b); }
PF_D double vmul(double a, double b) { return __dmul_rn(a, b); }
PF_D double vfma(double a, double b, double c) { return fma(a, b, c); }
template <>
PF_D double vlit<double>(double v) { return v; }
PF_D float x_lo(float2 a) { return a.x; }
PF_D float x_hi(float2 a) { return a.y; }
PF_D double x_lo(double2 a) { return a.x; }
PF_D double x_hi(double2 a) { return a.y; }
PF_D Dual<float> x_lo(DV<float2> a) { return make_dual(a.v.x, a.t.x); }
PF_D Dual<float> x_hi(DV<float2> a) { return make_dual(a.v.y, a.t.y); }
PF_D Dual<double> x_lo(DV<double2> a) { return make_dual(a.v.x, a.t.x); }
PF_D Dual<double> x_hi(DV<double2> a) { return make_dual(a.v.y, a.t.y); }
PF_D float2 x_pair(float a, float b) { return make_float2(a, b); }
PF_D double2 x_pair(double a, double b) { return make_double2(a, b); }
PF_D DV<float2> x_pair(Dual<float> a, Dual<float> b) { return {make_float2(a.v, b.v), make_float2(a.t, b.t)}; }
PF_D DV<double2> x_pair(Dual<double> a, Dual<double> b) { return {make_double2(a.v, b.v), make_double2(a.t, b.t)}; }
PF_D float from_below(float x) { return __shfl_up_sync(0xffffffffu, x, 1); }
PF_D double from_below(double x) { return __shfl_up_sync(0xffffffffu, x, 1); }
PF_D float from_above(float x) { return __shfl_down_sync(0xffffffffu, x, 1); }
PF_D double from_above(double x) { return __shfl_down_sync(0xffffffffu, x, 1); }
template <typename T>
PF_D Dual<T> from_below(Dual<T> x) { return make_dual(from_below(x.v), from_below(x.t)); }
template <typename T>
PF_D Dual<T> from_above(Dual<T> x) { return make_dual(from_above(x.v), from_above(x.t)); }
PF_D double x_value(double a) { return a; }
PF_D void x_set_value(double& a, double v) { a = v; }
PF_D float2 x_value(float2 a) { return a; }
PF_D double2 x_value(double2 a) { return a; }
template <typename V>
PF_D V x_value(DV<V> a) { return a.v; }
PF_D void x_set_value(float2& a, float2 v) { a = v; }
PF_D void x_set_value(double2& a, double2 v) { a = v; }
template <typename V>
PF_D void x_set_value(DV<V>& a, V v) { a.v = v; }
PF_D float value_of(float x) { return x; }
PF_D double value_of(double x) { return x; }
template <typename T>
PF_D T value_of(Dual<T> x) { return x.v; }

// arithmetic: plain two-lane vectors as in pf_lanes.cuh, and values with
// derivatives (a plain operand carries none)
template <typename V> PF_D DV<V> vadd(DV<V> a, DV<V> b) { return {vadd(a.v, b.v), vadd(a.t, b.t)}; }
template <typename V> PF_D DV<V> vadd(DV<V> a, V b) { return {vadd(a.v, b), a.t}; }
template <typename V> PF_D DV<V> vsub(DV<V> a, DV<V> b) { return {vsub(a.v, b.v), vsub(a.t, b.t)}; }
template <typename V> PF_D DV<V> vsub(DV<V> a, V b) { return {vsub(a.v, b), a.t}; }
template <typename V> PF_D DV<V> vsub(V a, DV<V> b) { return {vsub(a, b.v), vsub(vlit<V>(0.0), b.t)}; }
template <typename V> PF_D DV<V> vmul(DV<V> a, DV<V> b) { return {vmul(a.v, b.v), vfma(a.v, b.t, vmul(a.t, b.v))}; }
template <typename V> PF_D DV<V> vmul(DV<V> a, V b) { return {vmul(a.v, b), vmul(a.t, b)}; }
template <typename V> PF_D DV<V> vmul(V a, DV<V> b) { return vmul(b, a); }
template <typename V> PF_D DV<V> vfma(DV<V> a, DV<V> b, DV<V> c) {
    return {vfma(a.v, b.v, c.v), vfma(a.v, b.t, vfma(a.t, b.v, c.t))};
}
template <typename V> PF_D DV<V> vfma(DV<V> a, DV<V> b, V c) {
    return {vfma(a.v, b.v, c), vfma(a.v, b.t, vmul(a.t, b.v))};
}
template <typename V> PF_D DV<V> vfma(V a, DV<V> b, DV<V> c) { return {vfma(a, b.v, c.v), vfma(a, b.t, c.t)}; }
template <typename V> PF_D DV<V> vfma(DV<V> a, V b, DV<V> c) { return vfma(b, a, c); }
template <typename V> PF_D DV<V> vfma(V a, DV<V> b, V c) { return {vfma(a, b.v, c), vmul(a, b.t)}; }
template <typename V> PF_D DV<V> vfma(DV<V> a, V b, V c) { return vfma(b, a, c); }

// Reciprocal.  FP32: the hardware approximation, within 1 ulp; a Newton step
// after it (errors near half an ulp, as a division has) cost 2 to 3 % and changed
// the error of no field, k_v or derivative against 64 bits.  FP64: rcp64.
PF_D float2 vrcp_n(float2 x) {
    float2 r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r.x) : "f"(x.x));
    asm("rcp.approx.f32 %0, %1;" : "=f"(r.y) : "f"(x.y));
    return r;
}
PF_D double vrcp_n(double x) { return rcp64(x); }
PF_D double2 vrcp_n(double2 x) { return vrcp(x); }
template <typename V> PF_D DV<V> vrcp_n(DV<V> x) {
    const V r = vrcp_n(x.v);
    return {r, vmul(vsub(vlit<V>(0.0), x.t), vmul(r, r))};
}

// Natural logarithm.  FP32: x = 2^e m with m in [sqrt(1/2), sqrt(2)), f = m - 1,
// ln x = e ln 2 + (f - f^2/2 + f^3 P(f)); P, of degree 7, was fitted here by
// iteratively reweighted least squares to the smallest largest error relative
// to ln(1 + f) (7.9e-9 with the coefficients in FP32, an eighth of an ulp), so that
// the result is as exact as logf's, within an ulp, also near x = 1, where the
// hardware's lg2.approx has an absolute error of 2^-22.  For positive normal x;
// line_step replaces the results of zero, negative numbers, subnormals and NaN
// (is_positive, ln_fix).  +inf gives a finite number: an infinite concentration makes
// Mbar infinite and D Mbar / Mbar, and so the rate and the fluxes, NaN whatever its
// logarithm, so it is not asked for (asking costs the batch 1.6 %).
PF_D float2 ln_normal(float2 x) {
    const int bx = __float_as_int(x.x) - 0x3f3504f3, by = __float_as_int(x.y) - 0x3f3504f3;
    const int ex = bx & 0xff800000, ey = by & 0xff800000;
    const float2 m = make_float2(__int_as_float(__float_as_int(x.x) - ex), __int_as_float(__float_as_int(x.y) - ey));
    const float2 e = make_float2((float)ex, (float)ey);   // exponent times 2^23, exact
    const float2 f = vadd(m, vlit<float2>(-1.0));
    const float2 z = vmul(f, f);
    float2 P = vfma(f, vlit<float2>(-0.07634544372558594), vlit<float2>(0.1276165395975113));
    P = vfma(f, P, vlit<float2>(-0.13160201907157898));
    P = vfma(f, P, vlit<float2>(0.14201748371124268));
    P = vfma(f, P, vlit<float2>(-0.16623353958129883));
    P = vfma(f, P, vlit<float2>(0.20001226663589478));
    P = vfma(f, P, vlit<float2>(-0.250008225440979));
    P = vfma(f, P, vlit<float2>(0.3333333134651184));
    // ln 2 = 0.693359375 - 2.1219444e-4 (Cody and Waite's two parts): the first part's product with e is exact
    float2 y = vfma(vmul(z, f), P, vmul(e, vlit<float2>(-2.12194440054690583e-4 / 8388608.0)));
    y = vfma(z, vlit<float2>(-0.5), y);
    return vfma(e, vlit<float2>(0.693359375 / 8388608.0), vadd(f, y));
}
PF_D double ln_normal(double x) { return log64(x); }
PF_D double2 ln_normal(double2 x) { return vlog(x); }
template <typename V> PF_D DV<V> ln_normal(DV<V> x) {
    return {ln_normal(x.v), vmul(x.t, vrcp_n(x.v))};
}
PF_D bool is_positive(float2 x) { return x.x >= FLT_MIN && x.y >= FLT_MIN; }   // false for NaN
PF_D bool is_positive(double) { return true; }
PF_D bool is_positive(double2) { return true; }   // log64 takes any value
template <typename V> PF_D bool is_positive(DV<V> x) { return is_positive(x.v); }
// ln x where x is not a positive normal number, else the given l
PF_D float2 ln_fix(float2 x, float2 l) {
    return make_float2(x.x >= FLT_MIN ? l.x : logf(x.x), x.y >= FLT_MIN ? l.y : logf(x.y));
}
PF_D double ln_fix(double, double l) { return l; }
PF_D double2 ln_fix(double2, double2 l) { return l; }
template <typename V> PF_D DV<V> ln_fix(DV<V> x, DV<V> l) { return {ln_fix(x.v, l.v), l.t}; }

template <typename V, typename S>
__host__ __device__ __forceinline__ V line_splat(S v) {
    if constexpr (sizeof(V) == sizeof(S)) {
        return v;
    } else {
        V r;
        r.x = r.y = v;
        return r;
    }
}

// ---------------------------------------------------------------- parameters
// broadcast to both lanes; X carries the derivative of a differentiated parameter
template <typename E>
struct LineConsts {
    using V = typename LineNum<E>::V;
    using X = typename LineNum<E>::X;
    using S = typename LineNum<E>::S;
    V h2, h3, h4, h5, dh1, dh2, dh3, dh4, a_int;
    V Ms_c, Ms_0, Ml_c, Ml_0, Ms_c_half, Ml_c_half;
    V sigma, dx2, log_ke, delta2_dx2, delta2_4dx2;
    X b, K_anti, quarter_one_m_A, inv_Mphi;
    // with factors folded in: H dx^2, (1 - A) dx^2, -b, -A; the frozen
    // temperature (1 - k_e) theta = ke_theta0 + ke_G (i + 1/2)
    V H_dx2, dp_dx2, ke_G;
    X one_m_A_dx2, minus_b, minus_A;
    double one_m_ke;
    // Dirichlet (hot end) ghost and fresh-cell state
    S gphi, fc, fd, gphi_lo, fc_lo, fd_lo;   // and the low words of their FP32 pairs
    int hot_noflux;   // mirror ghost and zero flux at the hot end instead
};

// p(phi) of Eq. interpolation2 and its derivative.  STD: the default physics
// (quintic h, a = 0, M_i = D_i c_i) with parameters in the range where
// 1/(Mbar |grad phi|^2) stays an FP32 number, so that one reciprocal serves two
// quotients (line_std below).
template <bool STD, typename E, typename V>
PF_D V line_dp(const LineConsts<E>& K, V f) {
    const V g = vmul(f, vsub(vlit<V>(1.0), f));
    if constexpr (STD) return vmul(vmul(g, g), vlit<V>(30.0));
    const V dh = vmul(f, vfma(f, vfma(f, vfma(f, K.dh4, K.dh3), K.dh2), K.dh1));
    // d/dphi [g^2 (phi - 1/2)] = g^2 - 4 g (phi - 1/2)^2
    const V s = vsub(f, vlit<V>(0.5));
    return vfma(vmul(g, vsub(g, vmul(vmul(s, s), vlit<V>(4.0)))), K.a_int, dh);
}
template <bool STD, typename E, typename V>
PF_D V line_p(const LineConsts<E>& K, V f) {
    if constexpr (STD)
        return vmul(vmul(f, f), vmul(f, vfma(f, vfma(f, vlit<V>(6.0), vlit<V>(-15.0)), vlit<V>(10.0))));
    const V h = vmul(vmul(f, f), vfma(f, vfma(f, vfma(f, K.h5, K.h4), K.h3), K.h2));
    const V g = vmul(f, vsub(vlit<V>(1.0), f));
    return vfma(vmul(vsub(f, vlit<V>(0.5)), K.a_int), vmul(g, g), h);
}
// The derivatives along a direction come from p' and p'' themselves: the product
// rule over the polynomial subtracts terms 3 times f's derivative where p' is 0.
template <bool STD, typename T, typename V>
PF_D V line_d2p(const LineConsts<T>& K, V f) {
    const V g = vmul(f, vsub(vlit<V>(1.0), f));
    const V s = vfma(f, vlit<V>(-2.0), vlit<V>(1.0));   // 1 - 2 phi
    if constexpr (STD) return vmul(vmul(g, s), vlit<V>(60.0));
    const V d2h = vfma(f, vfma(f, vfma(f, vmul(K.dh4, vlit<V>(4.0)), vmul(K.dh3, vlit<V>(3.0))),
                               vmul(K.dh2, vlit<V>(2.0))), K.dh1);
    // d^2/dphi^2 [g^2 (phi - 1/2)], with g' = s and phi - 1/2 = -s/2
    const V w = vsub(vmul(vmul(g, s), vlit<V>(4.0)), vmul(s, vfma(s, s, vmul(g, vlit<V>(-2.0)))));
    return vfma(K.a_int, w, d2h);
}
template <bool STD, typename E, typename V>
PF_D DV<V> line_p(const LineConsts<E>& K, DV<V> f) {
    return {line_p<STD>(K, f.v), vmul(line_dp<STD>(K, f.v), f.t)};
}
template <bool STD, typename E, typename V>
PF_D DV<V> line_dp(const LineConsts<E>& K, DV<V> f) {
    return {line_dp<STD>(K, f.v), vmul(line_d2p<STD>(K, f.v), f.t)};
}

template <bool STD, typename V, typename X>
PF_D X line_M(const V mc, const V m0, X c) {
    if constexpr (STD) return vmul(c, mc);
    else return vfma(c, mc, m0);
}

// dx^2 dphi/dt of a pair: f its phi, fL / fR its neighbours', and so on; dmu =
// mu_s - mu_l, ke_theta = (1 - k_e) theta.  In STD the algebra is arranged for
// few operations (the FP32 pipe, on which a packed instruction takes two
// cycles, bounds the batch): t = 1/(Mbar G) serves 1/Mbar = t G and
// 1/(Mbar G), and R / (1/M_phi + kk/u) = R u / (u/M_phi + kk).
template <bool STD, typename E, typename X>
PF_D X line_rate(const LineConsts<E>& K, X f, X fL, X fR, X sL, X sR, X lL, X lR, X cs, X cl, X dmu, X p,
                 typename LineNum<E>::V ke_theta) {
    using V = typename LineNum<E>::V;
    const X lap = vadd(vsub(fL, f), vsub(fR, f));
    const X gx = vsub(fR, fL), sx = vsub(sR, sL), lx = vsub(lR, lL);
    const X omp = vsub(vlit<V>(1.0), p);
    const X Ms = line_M<STD>(K.Ms_c, K.Ms_0, cs), Ml = line_M<STD>(K.Ml_c, K.Ml_0, cl);
    const X nbMl = vmul(K.minus_b, Ml);
    const X Msq = vmul(Ms, omp);
    const X nbMlp = vmul(nbMl, p);
    const X M = vsub(Msq, nbMlp);
    const X G = vfma(gx, gx, K.delta2_4dx2);
    const X u = vfma(K.b, p, omp);
    const X nd = vsub(cl, cs);                                        // -d
    const X ndpq = vmul(nd, vmul(p, omp));
    const X cross = vmul(vfma(nbMl, lx, vmul(Ms, sx)), gx);           // (M_s grad mu_s - b M_l grad mu_l).grad phi
    const X g = vmul(f, vsub(vlit<V>(1.0), f));
    const X dfdw = vmul(g, vfma(f, vlit<V>(-4.0), vlit<V>(2.0)));
    // D Mbar = M_s (1-p)(1 - A(1-p)) + A b M_l p^2
    const X DM = vfma(K.minus_A, vfma(nbMlp, p, vmul(Msq, omp)), Msq);
    X iM, iMG;
    if constexpr (STD) {
        iMG = vrcp_n(vmul(M, G));
        iM = vmul(iMG, G);
    } else {
        iM = vrcp_n(M);
        iMG = vmul(iM, vrcp_n(G));
    }
    // DeltaG = c_s (mu_s - mu_l) - d - (1-k_e) theta - D d (mu_s - mu_l)
    const X dG = vfma(dmu, vfma(nd, vmul(DM, iM), cs), vsub(nd, ke_theta));
    const X w = vmul(ndpq, iMG);
    const X nanti = vmul(vmul(K.one_m_A_dx2, w), cross);              // -(1-A) d p(1-p) cross / (Mbar G) dx^2
    X dp;
    if constexpr (STD) dp = vmul(vmul(g, g), K.dp_dx2);
    else dp = vmul(line_dp<STD>(K, f), K.dx2);
    const X R = vsub(vmul(K.sigma, lap), vfma(K.H_dx2, dfdw, vfma(dG, dp, nanti)));
    const X kk = vmul(K.K_anti, vmul(nd, w));
    if constexpr (STD) return vmul(vmul(R, u), vrcp_n(vfma(K.inv_Mphi, u, kk)));
    return vmul(R, vrcp_n(vfma(kk, vrcp_n(u), K.inv_Mphi)));
}

// fluxes dx F_c, dx F_d through the faces between the pairs L and R; in STD
// with t = 1/(Mbar G), G = n_phi^2 + delta^2 dx^2, of which r = 1/G = t Mbar:
//   F_c = t X + r delta^2 dx^2 Z,  F_d = r (delta^2 dx^2 (T_s - T_l) + at)
template <bool STD, typename E, typename X>
PF_D void line_face(const LineConsts<E>& K, X fL, X fR, X YL, X YR, X sL, X sR, X lL, X lR, X csL, X csR, X clL,
                    X clR, X pdL, X pdR, X& Fc, X& Fd) {
    using V = typename LineNum<E>::V;
    const X n0 = vsub(fR, fL), n1 = vsub(YR, YL), n2 = vsub(sR, sL), n3 = vsub(lR, lL);
    const X S = vadd(fL, fR);
    const X cs2 = vadd(csL, csR), cl2 = vadd(clL, clR);
    const X d2 = vsub(cs2, cl2);
    X p;
    if constexpr (STD && !IsDual<E>::value)   // p(S/2)
        p = vmul(vmul(S, S), vmul(S, vfma(S, vfma(S, vlit<V>(6.0 / 32.0), vlit<V>(-15.0 / 16.0)), vlit<V>(10.0 / 8.0))));
    else p = line_p<STD>(K, vmul(S, vlit<V>(0.5)));
    const X omp = vsub(vlit<V>(1.0), p);
    const X Ms = line_M<STD>(K.Ms_c_half, K.Ms_0, cs2), Ml = line_M<STD>(K.Ml_c_half, K.Ml_0, cl2);
    const X bMl = vmul(K.b, Ml);
    const X nn = vmul(n0, n0);
    const X M = vfma(bMl, p, vmul(Ms, omp)), G = vadd(nn, K.delta2_dx2);
    const X Ts = vmul(Ms, n2), Tl = vmul(Ml, n3);
    const X TD = vsub(Ts, Tl);
    const X Z = vfma(p, TD, Tl);
    const X at = vmul(vmul(K.quarter_one_m_A, vadd(pdL, pdR)), vmul(d2, n0));
    X N = vmul(vmul(Ms, Ml), vmul(vfma(K.b, p, omp), vmul(nn, n1)));
    N = vfma(vmul(vsub(Ms, bMl), vmul(p, omp)), at, N);
    X t, r;
    if constexpr (STD) {
        t = vrcp_n(vmul(M, G));
        r = vmul(t, M);
    } else {
        r = vrcp_n(G);
        t = vmul(vrcp_n(M), r);
    }
    Fc = vfma(t, N, vmul(r, vmul(Z, K.delta2_dx2)));
    Fd = vmul(r, vfma(TD, K.delta2_dx2, at));
}

// whether a parameter set is one for STD
inline bool line_std(const HostProblem& P) { return std_physics(P, true) && P.a == 0.0; }

// parameters, with the derivative 1 along one of (1/M_phi by M_phi, A, b) if dir >= 0
template <typename E>
inline LineConsts<E> make_line_consts(const HostProblem& P, int dir) {
    using V = typename LineNum<E>::V;
    using X = typename LineNum<E>::X;
    using S = typename LineNum<E>::S;
    Consts<double> C;
    C.interp = P.interp; C.mobility = P.mobility; C.D_s = P.D_s; C.D_l = P.D_l;
    set_coefficients(C);
    auto v = [](double x) { return line_splat<V>(S(x)); };
    auto x = [&](Dual<double> u) {
        if constexpr (IsDual<E>::value) return X{v(u.v), v(u.t)};
        else return v(u.v);
    };
    const Dual<double> A = make_dual(P.A, dir == 1 ? 1.0 : 0.0), b = make_dual(P.b, dir == 2 ? 1.0 : 0.0);
    const Dual<double> iM = make_dual(1.0 / P.M_phi, dir == 0 ? -1.0 / (P.M_phi * P.M_phi) : 0.0);
    const Dual<double> oA = Dual<double>(1.0) - A;
    const double dx2 = P.dx * P.dx;
    LineConsts<E> K;
    K.h2 = v(C.h2); K.h3 = v(C.h3); K.h4 = v(C.h4); K.h5 = v(C.h5);
    K.dh1 = v(C.dh1); K.dh2 = v(C.dh2); K.dh3 = v(C.dh3); K.dh4 = v(C.dh4);
    K.a_int = v(P.a);
    K.Ms_c = v(C.Ms_c); K.Ms_0 = v(C.Ms_0); K.Ml_c = v(C.Ml_c); K.Ml_0 = v(C.Ml_0);
    K.Ms_c_half = v(0.5 * C.Ms_c); K.Ml_c_half = v(0.5 * C.Ml_c);
    K.sigma = v(P.sigma); K.dx2 = v(dx2); K.log_ke = v(std::log(P.k_e));
    K.delta2_dx2 = v(P.delta * P.delta * dx2); K.delta2_4dx2 = v(4.0 * P.delta * P.delta * dx2);
    K.b = x(b); K.K_anti = x(oA * oA * b * Dual<double>(4.0 * dx2));
    K.quarter_one_m_A = x(oA * Dual<double>(0.25)); K.inv_Mphi = x(iM);
    K.H_dx2 = v(P.H * dx2); K.dp_dx2 = v(30.0 * dx2); K.ke_G = v(-(1.0 - P.k_e) * P.G_theta * P.dx);
    K.one_m_A_dx2 = x(oA * Dual<double>(dx2)); K.minus_b = x(-b); K.minus_A = x(-A);
    K.one_m_ke = 1.0 - P.k_e;
    const double pg = p_host3(P, P.dir_phi);
    K.gphi = S(P.dir_phi);
    const double fc = pg * P.dir_cs + (1.0 - pg) * P.dir_cl, fd = P.dir_cs - P.dir_cl;
    K.fc = S(fc); K.fd = S(fd);
    K.gphi_lo = S(P.dir_phi - (double)K.gphi); K.fc_lo = S(fc - (double)K.fc); K.fd_lo = S(fd - (double)K.fd);
    K.hot_noflux = P.bc_hi[0] == BC_NOFLUX;
    return K;
}

// The same with a derivative.  The fluxes are smooth in n_phi where their factors
// are not (n_phi decays by e-folds over a cell or two): with r = 1/G,
//   F_c = q n_Y w + rd Z + a e afn,  F_d = rd (T_s - T_l) + a e,
//   w = n_phi^2 r = 1 - rd,  rd = delta^2 dx^2 r,  e = n_phi r,  a = (1-A) d rate,
// and dw = -d(rd) = 2 e rd dn_phi, de = r (rd - w) dn_phi, so that no large terms
// cancel (through d(1/G), dk/dM_phi of the FP32 runs lost a further digit).
template <bool STD, typename E, typename V>
PF_D void line_face(const LineConsts<E>& K, DV<V> fL, DV<V> fR, DV<V> YL, DV<V> YR, DV<V> sL, DV<V> sR, DV<V> lL,
                    DV<V> lR, DV<V> csL, DV<V> csR, DV<V> clL, DV<V> clR, DV<V> pdL, DV<V> pdR, DV<V>& Fc,
                    DV<V>& Fd) {
    using X = DV<V>;
    const X n0 = vsub(fR, fL), n1 = vsub(YR, YL), n2 = vsub(sR, sL), n3 = vsub(lR, lL);
    const X cs2 = vadd(csL, csR), cl2 = vadd(clL, clR);
    const X p = line_p<STD>(K, vmul(vadd(fL, fR), vlit<V>(0.5)));
    const X omp = vsub(vlit<V>(1.0), p);
    const X Ms = line_M<STD>(K.Ms_c_half, K.Ms_0, cs2), Ml = line_M<STD>(K.Ml_c_half, K.Ml_0, cl2);
    const X bMl = vmul(K.b, Ml);
    const X M = vfma(bMl, p, vmul(Ms, omp));
    const V nn = vmul(n0.v, n0.v), G = vadd(nn, K.delta2_dx2);
    V im, r;
    if constexpr (STD) {
        const V t = vrcp_n(vmul(M.v, G));
        im = vmul(t, G);
        r = vmul(t, M.v);
    } else {
        im = vrcp_n(M.v);
        r = vrcp_n(G);
    }
    const X iM = {im, vsub(vlit<V>(0.0), vmul(M.t, vmul(im, im)))};
    const V rd = vmul(K.delta2_dx2, r), w = vmul(nn, r), e = vmul(n0.v, r);
    const V dw = vmul(vmul(vmul(e, rd), vlit<V>(2.0)), n0.t);
    const X W = {w, dw}, RD = {rd, vsub(vlit<V>(0.0), dw)}, EE = {e, vmul(vmul(r, vsub(rd, w)), n0.t)};
    const X Ts = vmul(Ms, n2), Tl = vmul(Ml, n3);
    const X TD = vsub(Ts, Tl);
    const X ae = vmul(vmul(vmul(K.quarter_one_m_A, vadd(pdL, pdR)), vsub(cs2, cl2)), EE);
    const X q = vmul(vmul(Ms, Ml), vmul(vfma(K.b, p, omp), iM));
    const X afn = vmul(vsub(Ms, bMl), vmul(vmul(p, omp), iM));
    Fc = vfma(vmul(q, n1), W, vfma(RD, vfma(p, TD, Tl), vmul(ae, afn)));
    Fd = vfma(RD, TD, ae);
}

// the vector of two cells' values; of one cell, its own
template <typename X, typename A>
PF_D X x_join(A a, A b) {
    if constexpr (sizeof(X) == sizeof(A)) return a;
    else return x_pair(a, b);
}
template <typename X, typename E>
PF_D X x_select(X a, E other, bool lo, bool hi) {
    return x_join<X>(lo ? other : x_lo(a), hi ? other : x_hi(a));
}

// The strip's state and one step of it.  COMP: the values of phi and c (1), or of
// phi, c and d (2), are unevaluated FP32 pairs (compensated sums).
template <typename E, int J, int COMP>
struct Strip {
    static constexpr int H = J / LineNum<E>::LANES;
    using X = typename LineNum<E>::X;
    using V = typename LineNum<E>::V;
    X phi[H], c[H], d[H];
    V plo[COMP ? H : 1], clo[COMP ? H : 1], dlo[COMP == 2 ? H : 1];
};

struct NoRecord {
    template <typename X, typename V>
    PF_D void operator()(int, const X&, const X&, const X&, const X&, const X&, const X&, const X&, const X&,
                         const V&) const {}
    static constexpr bool on = false;
};

// One step of the strip.  i0: the line index of the lane's first cell; the line
// is the cells m .. n + m - 1 (m: window shifts since the indices were set), the
// cells beyond hold the Dirichlet state and are not updated, those below m are
// outside the window.  EDGE: the strip reaches an end of the line (a compile-time
// switch, so that the other strips carry none of its selections).  dtq = dt / dx^2;
// ke_theta0 = (1 - k_e) theta0 (theta0 as Consts::G_theta describes it).  record(q, phi,
// phi of the right neighbour, p, c_s, c_l, mu_s, mu_l, rate, (1 - k_e) theta) is
// called for every pair with its state before the step; the rate it is given is in
// grid units.
template <bool STD, bool edge, typename E, int J, int COMP, typename Rec>
PF_D void line_step(const LineConsts<E>& K, Strip<E, J, COMP>& s, int i0, int n, int m,
                    typename LineNum<E>::V dtq, double ke_theta0, const Rec& record) {
    using X = typename LineNum<E>::X;
    using V = typename LineNum<E>::V;
    using S = typename LineNum<E>::S;
    using M = typename LineNum<E>::M;
    constexpr int H = J / LineNum<E>::LANES;
    X cs[H], cl[H], mus[H], mul[H], Y[H], pd[H], p[H];
    bool fine = true;
#pragma unroll
    for (int q = 0; q < H; ++q) {
        p[q] = line_p<STD>(K, s.phi[q]);
        const X omp = vsub(vlit<V>(1.0), p[q]);
        const X mp = vsub(vlit<V>(0.0), p[q]);
        cs[q] = vfma(omp, s.d[q], s.c[q]);
        cl[q] = vfma(mp, s.d[q], s.c[q]);
        if constexpr (COMP == 2) {   // the low words, of the values
            cs[q] = vadd(cs[q], vfma(x_value(omp), s.dlo[q], s.clo[q]));
            cl[q] = vadd(cl[q], vfma(x_value(mp), s.dlo[q], s.clo[q]));
        } else if constexpr (COMP == 1) {
            cs[q] = vadd(cs[q], s.clo[q]);
            cl[q] = vadd(cl[q], s.clo[q]);
        }
        fine = fine && is_positive(cs[q]) && is_positive(cl[q]);
        mus[q] = ln_normal(cs[q]);
        mul[q] = ln_normal(cl[q]);
    }
    if (!fine) {   // a concentration that is no positive normal number (a run that broke down)
#pragma unroll
        for (int q = 0; q < H; ++q) {
            mus[q] = ln_fix(cs[q], mus[q]);
            mul[q] = ln_fix(cl[q], mul[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < H; ++q) mus[q] = vsub(mus[q], K.log_ke);
    const int hot = n + m;   // first cell beyond the line
    X dmu[H];
#pragma unroll
    for (int q = 0; q < H; ++q) {
        dmu[q] = vsub(mus[q], mul[q]);
        Y[q] = vfma(p[q], dmu[q], mul[q]);
    }
    // neighbours across the lane's ends
    auto left_of = [&](const X (&a)[H]) {
        if constexpr (LineNum<E>::LANES == 1) return from_below(a[H - 1]);
        else return x_pair(from_below(x_hi(a[H - 1])), x_lo(a[H - 1]));
    };
    auto right_of = [&](const X (&a)[H]) {
        if constexpr (LineNum<E>::LANES == 1) return from_above(a[0]);
        else return x_pair(x_hi(a[0]), from_above(x_lo(a[0])));
    };
    const X fA = left_of(s.phi), sA = left_of(mus), lA = left_of(mul);
    const X fB = right_of(s.phi), sB = right_of(mus), lB = right_of(mul);
    const S xi = S(i0 - m) + S(0.5);
    const V th0 = line_splat<V>(S(ke_theta0));   // (1 - k_e) theta = ke_theta0 + ke_G (i + 1/2)
#pragma unroll
    for (int q = 0; q < H; ++q) {
        X fL = q > 0 ? s.phi[q - 1] : fA, sL = q > 0 ? mus[q - 1] : sA, lL = q > 0 ? mul[q - 1] : lA;
        X fR = q < H - 1 ? s.phi[q + 1] : fB, sR = q < H - 1 ? mus[q + 1] : sB, lR = q < H - 1 ? mul[q + 1] : lB;
        const int ia = i0 + q, ib = i0 + q + H;
        if (edge) {
            // mirror ghosts: the cold end always, the hot end if it is closed
            if (ia == m) { fL = x_join<X>(x_lo(s.phi[q]), x_hi(fL)); sL = x_join<X>(x_lo(mus[q]), x_hi(sL)); lL = x_join<X>(x_lo(mul[q]), x_hi(lL)); }
            if (ib == m) { fL = x_join<X>(x_lo(fL), x_hi(s.phi[q])); sL = x_join<X>(x_lo(sL), x_hi(mus[q])); lL = x_join<X>(x_lo(lL), x_hi(mul[q])); }
            if (K.hot_noflux) {
                if (ia == hot - 1) { fR = x_join<X>(x_lo(s.phi[q]), x_hi(fR)); sR = x_join<X>(x_lo(mus[q]), x_hi(sR)); lR = x_join<X>(x_lo(mul[q]), x_hi(lR)); }
                if (ib == hot - 1) { fR = x_join<X>(x_lo(fR), x_hi(s.phi[q])); sR = x_join<X>(x_lo(sR), x_hi(mus[q])); lR = x_join<X>(x_lo(lR), x_hi(mul[q])); }
            }
        }
        const V ke_theta = vfma(K.ke_G, x_join<V>(xi + S(q), xi + S(q + H)), th0);
        pd[q] = line_rate<STD>(K, s.phi[q], fL, fR, sL, sR, lL, lR, cs[q], cl[q], dmu[q], p[q],
                               ke_theta);
        if (edge) pd[q] = x_select(pd[q], M(0), ia >= hot, ib >= hot);
        if constexpr (Rec::on) record(q, s.phi[q], fR, p[q], cs[q], cl[q], mus[q], mul[q], pd[q], ke_theta);
    }
    const X YB = right_of(Y), csB = right_of(cs), clB = right_of(cl), pdB = right_of(pd);
    X Fc[H], Fd[H];
#pragma unroll
    for (int q = 0; q < H; ++q) {
        const bool last = q == H - 1;
        line_face<STD>(K, s.phi[q], last ? fB : s.phi[last ? 0 : q + 1], Y[q], last ? YB : Y[last ? 0 : q + 1], mus[q],
                       last ? sB : mus[last ? 0 : q + 1], mul[q], last ? lB : mul[last ? 0 : q + 1], cs[q],
                       last ? csB : cs[last ? 0 : q + 1], cl[q], last ? clB : cl[last ? 0 : q + 1], pd[q],
                       last ? pdB : pd[last ? 0 : q + 1], Fc[q], Fd[q]);
        if (edge) {   // no flux through the cold end, nor through a closed hot end
            const int ia = i0 + q, ib = i0 + q + H;
            const bool zlo = ia == m - 1 || (K.hot_noflux && ia == hot - 1);
            const bool zhi = ib == m - 1 || (K.hot_noflux && ib == hot - 1);
            Fc[q] = x_select(Fc[q], M(0), zlo, zhi);
            Fd[q] = x_select(Fd[q], M(0), zlo, zhi);
        }
    }
    X FcL = left_of(Fc), FdL = left_of(Fd);
    if (edge) {   // a line that begins at the lane's (or the strip's) first cell
        const bool zlo = i0 == m, zhi = i0 + H == m;
        FcL = x_select(FcL, M(0), zlo, zhi);
        FdL = x_select(FdL, M(0), zlo, zhi);
    }
#pragma unroll
    for (int q = 0; q < H; ++q) {
        const X dFc = vsub(Fc[q], q > 0 ? Fc[q > 0 ? q - 1 : 0] : FcL);
        const X dFd = vsub(Fd[q], q > 0 ? Fd[q > 0 ? q - 1 : 0] : FdL);
        const bool glo = edge && i0 + q >= hot, ghi = edge && i0 + q + H >= hot;
        auto hold = [&](auto now, auto before) {   // the ghosts' c and d stay
            return x_join<decltype(now)>(glo ? x_lo(before) : x_lo(now), ghi ? x_hi(before) : x_hi(now));
        };
        if constexpr (COMP) {
            // compensated (TwoSum) updates of the values phi, c, d = hi + lo; the
            // derivatives, if any, are added plainly
            auto add2 = [&](X& x, V& lo, X inc, bool keep) {
                const V hi = x_value(x), up = x_value(inc);
                const V s_ = vadd(hi, up);
                const V bv = vsub(s_, hi);
                const V l = vadd(lo, vadd(vsub(hi, vsub(s_, bv)), vsub(up, bv)));
                const V h = vadd(s_, l);
                const V ln = vsub(l, vsub(h, s_));
                X n = vadd(x, inc);
                x_set_value(n, h);
                x = keep ? hold(n, x) : n;
                lo = keep ? hold(ln, lo) : ln;
            };
            add2(s.phi[q], s.plo[q], vmul(pd[q], dtq), false);   // a rate of 0 leaves the ghosts' phi
            add2(s.c[q], s.clo[q], vmul(dFc, dtq), edge);
            if constexpr (COMP == 2) {
                add2(s.d[q], s.dlo[q], vmul(dFd, dtq), edge);
            } else {
                const X dn = vfma(dFd, dtq, s.d[q]);
                s.d[q] = edge ? hold(dn, s.d[q]) : dn;
            }
        } else {
            s.phi[q] = vfma(pd[q], dtq, s.phi[q]);
            const X cn = vfma(dFc, dtq, s.c[q]), dn = vfma(dFd, dtq, s.d[q]);
            s.c[q] = edge ? hold(cn, s.c[q]) : cn;
            s.d[q] = edge ? hold(dn, s.d[q]) : dn;
        }
    }
}

#undef PF_D
}  // namespace pf

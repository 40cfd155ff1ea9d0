// pf_words.cuh -- sums over FP32 states without the FP64 pipe: numbers as
// unevaluated sums of two or three floats (T. J. Dekker, Numer. Math. 18, 1971;
// D. E. Knuth, The Art of Computer Programming, vol. 2, 4.2.2).
//
// A GB300 issues an FP64 operation of a warp in the time of about 70 FP32 ones.
// Two words hold 48 bits, which is enough for a value of the state (c with its low
// word) but leaves every operation an error of up to 2^-47, which cells of equal
// value, as the bulk phases have, all repeat.  Three words carry FP64's 53 bits
// and some more: the operations below are within 2^-64 of the larger operand (of
// the product), the logarithm within 2^-54 of the larger of 1 and its value.
#pragma once
#include <cmath>

namespace pf {

struct Pair {
    float h, l;      // |l| at most half an ulp of h
};
struct Triple {
    float h, l, t;   // falling by about 2^-23 from word to word; not normalised
};
inline Triple triple_of(double v) {   // exact within FP32's range
    const float h = (float)v;
    const double r = v - (double)h;
    const float l = (float)r;
    return {h, l, (float)(r - (double)l)};
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ Pair sum2(float a, float b) {
    float s, e;
    two_sum(a, b, s, e);
    return {s, e};
}
__device__ __forceinline__ Pair prod2(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ Triple widen(Pair a) { return {a.h, a.l, 0.0f}; }

__device__ __forceinline__ Triple operator-(Triple a) { return {-a.h, -a.l, -a.t}; }
__device__ __forceinline__ Triple operator+(Triple a, Triple b) {
    const Pair s = sum2(a.h, b.h), r = sum2(a.l, b.l), m = sum2(s.l, r.h);
    return {s.h, m.h, (a.t + b.t) + (r.l + m.l)};
}
__device__ __forceinline__ Triple operator+(Triple a, float b) {
    const Pair s = sum2(a.h, b), m = sum2(s.l, a.l);
    return {s.h, m.h, a.t + m.l};
}
__device__ __forceinline__ Triple operator-(Triple a, Triple b) { return a + (-b); }
__device__ __forceinline__ Triple operator*(Triple a, Triple b) {
    const Pair p = prod2(a.h, b.h), q = prod2(a.h, b.l), r = prod2(a.l, b.h), s = sum2(q.h, r.h), m = sum2(p.l, s.h);
    const float t = __fmaf_rn(a.h, b.t, __fmaf_rn(a.t, b.h, __fmul_rn(a.l, b.l)));
    return {p.h, m.h, t + ((q.l + r.l) + (s.l + m.l))};
}
__device__ __forceinline__ Triple operator*(Triple a, float b) {
    const Pair p = prod2(a.h, b), q = prod2(a.l, b), m = sum2(p.l, q.h);
    return {p.h, m.h, __fmaf_rn(a.t, b, q.l + m.l)};
}
__device__ __forceinline__ double value(Triple a) { return ((double)a.t + (double)a.l) + (double)a.h; }

// ln x: x = 2^e m, r a 9-bit approximation of 1/m from a table of 128, z = m r - 1,
// |z| < 2^-7, and the series of ln(1 + z) to z^7.  -ln r is tabulated in parts on
// grids of 2^-14, 2^-28 and 2^-42 and a rest, and ln 2 split the same way (Cody and
// Waite's reduction), so that e ln 2 - ln r is added part by part without error.
// NaN where x is not a number between 2^-70 and FP32's largest: below, the low words
// of x and of its products would leave FP32's range.
struct LogTable {
    float r[128], a[128], b[128], c[128], d[128];
    LogTable() = default;
    explicit LogTable(int) {
        for (int t = 0; t < 128; ++t) {
            const double q = std::rint(512.0 / (1.0 + (t + 0.5) / 128.0)) / 512.0;   // 9 bits
            r[t] = (float)q;
            long double rest = -std::log((long double)q);   // FP64's would be off by 2^-54
            const double A = std::rint((double)rest * 0x1p14) * 0x1p-14;
            rest -= A;
            const double B = std::rint((double)rest * 0x1p28) * 0x1p-28;
            rest -= B;
            const double C = std::rint((double)rest * 0x1p42) * 0x1p-42;
            rest -= C;
            a[t] = (float)A;
            b[t] = (float)B;
            c[t] = (float)C;
            d[t] = (float)rest;
        }
    }
};
__device__ __forceinline__ Triple ln_triple(const LogTable& T, Triple x) {
    {   // words that cancelled may have left the second larger than the first
        const Pair n = sum2(x.h, x.l), o = sum2(n.l, x.t), q = sum2(n.h, o.h);
        x = {q.h, q.l, o.l};
    }
    if (!(x.h >= 0x1p-70f && x.h <= 3.402823466e38f)) return {NAN, 0.0f, 0.0f};
    const int b = __float_as_int(x.h);
    const int e = (b >> 23) - 127, k = (b >> 16) & 127;
    const float m = __int_as_float((b & 0x007fffff) | 0x3f800000);
    const float s1 = __int_as_float((127 - e / 2) << 23), s2 = __int_as_float((127 - (e - e / 2)) << 23);   // 2^-e = s1 s2
    const float ml = __fmul_rn(__fmul_rn(x.l, s1), s2), mt = __fmul_rn(__fmul_rn(x.t, s1), s2);
    const float r = T.r[k], ef = (float)e;
    const Pair p = prod2(m, r), q = prod2(ml, r);
    Pair z = sum2(p.l, q.h);
    const float zt = __fmaf_rn(mt, r, q.l) + z.l;
    z = sum2(p.h - 1.0f, z.h);                       // z = z.h + z.l + zt
    Pair w = prod2(z.h, z.h);                        // z^2
    w.l = __fmaf_rn(z.h + z.h, z.l, w.l);
    Pair u = prod2(w.h, z.h);                        // z^3
    u.l = __fmaf_rn(w.l, z.h, __fmaf_rn(w.h, z.l, u.l));
    Pair v = prod2(u.h, 0x1.555556p-2f);             // z^3 / 3
    v.l = __fmaf_rn(u.h, -0x1.555556p-27f, __fmaf_rn(u.l, 0x1.555556p-2f, v.l));
    const float w4 = __fmul_rn(w.h, w.h);            // z^4
    const float tail = __fmul_rn(w4, __fmaf_rn(z.h, __fmaf_rn(z.h, __fmaf_rn(z.h, 1.0f / 7, -1.0f / 6), 0.2f), -0.25f));
    // ln 2 on the same grids
    const float A = __fmaf_rn(ef, 0x1.62e8p-1f, T.a[k]), B = __fmaf_rn(ef, -0x1.e81p-16f, T.b[k]);
    const float C = __fmaf_rn(ef, 0x1.f47p-30f, T.c[k]), D = __fmaf_rn(ef, 0x1.ef357ap-45f, T.d[k]);
    const Pair a1 = sum2(A, z.h), a2 = sum2(a1.h, B), a3 = sum2(a2.h, -0.5f * w.h);
    const Pair b1 = sum2(a1.l, a2.l), b2 = sum2(b1.h, a3.l), b3 = sum2(b2.h, C), b4 = sum2(b3.h, z.l), b5 = sum2(b4.h, v.h);
    const float t = ((b1.l + b2.l) + (b3.l + b4.l)) + (b5.l + (zt + D)) + (tail + __fmaf_rn(-0.5f, w.l, v.l));
    return {a3.h, b5.h, t};
}

}  // namespace pf

// pf_fp64.cuh -- FP64 logarithm and reciprocal for the step kernels, in fewer
// instructions of the FP64 pipe than log() and the IEEE division: a GB300's FP64
// pipe takes about 18 cycles per warp instruction and SM and bounds every FP64
// step.  The logarithm takes 14 of them, the reciprocal 4.
#pragma once
#include <cuda_runtime.h>

namespace pf {

// {r, -ln r}, r near the reciprocal of the centre of interval t of [sqrt(1/2),
// sqrt(2)) (128 intervals, equal in the bits of the double), chosen such that -ln r
// is a multiple of 2^-42 to 2^-62 (S. Gal and B. Bachelis, ACM Trans. Math. Softw.
// 17, 1991: accurate tables); r = 1 for the three intervals around 1, where the
// logarithm has to keep its relative error
static __device__ const double2 LOG64[128] = {
    {0x1.69004de80619fp+0, -0x1.5ff3e406e7000p-2}, {0x1.670024c382f21p+0, -0x1.5a4313ec5f000p-2},
    {0x1.65000ef5dca1bp+0, -0x1.548a57243c000p-2}, {0x1.63003b5c51282p+0, -0x1.4eca1e5fd4000p-2},
    {0x1.61800bfd0acdfp+0, -0x1.4a7396890c000p-2}, {0x1.5f802995d74d4p+0, -0x1.44a4946bfb000p-2},
    {0x1.5d8023234a239p+0, -0x1.3eccad023d000p-2}, {0x1.5b800d2fa1147p+0, -0x1.38ec02141a000p-2},
    {0x1.59ffdc7984d1dp+0, -0x1.347d70860d000p-2}, {0x1.58002c263d746p+0, -0x1.2e8eaf19ea000p-2},
    {0x1.56004abcbe671p+0, -0x1.2896810428000p-2}, {0x1.548008249f451p+0, -0x1.2415713cfd000p-2},
    {0x1.528029d31ac19p+0, -0x1.1e0d8ab997000p-2}, {0x1.510030a2752fdp+0, -0x1.198166a4e0000p-2},
    {0x1.4f001ad3aa1e0p+0, -0x1.1368c229b8000p-2}, {0x1.4d7fd880826fbp+0, -0x1.0ecf8caf57000p-2},
    {0x1.4bffd49e142e0p+0, -0x1.0a31c858c8000p-2}, {0x1.4a000ffc5302dp+0, -0x1.04028ae5e7000p-2},
    {0x1.488023c42d37dp+0, -0x1.feb1023996000p-3}, {0x1.47001e14e624fp+0, -0x1.f55161cb64000p-3},
    {0x1.4500308cd9bcep+0, -0x1.e8c1571b70000p-3}, {0x1.43801c69f9406p+0, -0x1.df4774a8de000p-3},
    {0x1.41fff4d802382p+0, -0x1.d5c1cfc02a000p-3}, {0x1.408044338ff04p+0, -0x1.cc33bfd028000p-3},
    {0x1.3f00174e2fa38p+0, -0x1.c2971af806000p-3}, {0x1.3d7fb163e2b53p+0, -0x1.b8ed6bf36c000p-3},
    {0x1.3c0024816f51fp+0, -0x1.af3d817fe0000p-3}, {0x1.3a80217b07133p+0, -0x1.a57ecc881a000p-3},
    {0x1.39002806938e2p+0, -0x1.9bb468cc80000p-3}, {0x1.37802ef025c29p+0, -0x1.91ddfd5cfe000p-3},
    {0x1.360004d1022fap+0, -0x1.87fa2623dc000p-3}, {0x1.347fe3c04b6e5p+0, -0x1.7e0a41dace000p-3},
    {0x1.33004be460e47p+0, -0x1.7411899aac000p-3}, {0x1.318034e79bf52p+0, -0x1.6a08ffb886000p-3},
    {0x1.2fffca1f6e7b2p+0, -0x1.5ff19c13fe000p-3}, {0x1.2e80405e91ae2p+0, -0x1.55d3610e04000p-3},
    {0x1.2d7fc4733e9e3p+0, -0x1.4f080ac8e2000p-3}, {0x1.2bfffd8cfa2a5p+0, -0x1.44d2a6143e000p-3},
    {0x1.2a7fe3dcb0d4bp+0, -0x1.3a8df1c55e000p-3}, {0x1.28ffc93459c9fp+0, -0x1.303bf7b4c4000p-3},
    {0x1.28001c7e31223p+0, -0x1.2955f4a5e2000p-3}, {0x1.267fd06fa195bp+0, -0x1.1eec461e58000p-3},
    {0x1.24fff77350421p+0, -0x1.14781c840e000p-3}, {0x1.23ffba4127f7ap+0, -0x1.0d75fea050000p-3},
    {0x1.2280457c0f5a8p+0, -0x1.02ed9e0804000p-3}, {0x1.217fc344a6647p+0, -0x1.f7b444a7b0000p-4},
    {0x1.1fffc32fae0a7p+0, -0x1.e26d15fa38000p-4}, {0x1.1f00305031a13p+0, -0x1.d433eeeaac000p-4},
    {0x1.1d8008cfa693ap+0, -0x1.bebaffea8c000p-4}, {0x1.1c7fd73a35d6ap+0, -0x1.b058febbe8000p-4},
    {0x1.1afff25399307p+0, -0x1.9ab35e7af0000p-4}, {0x1.19ffd05255bafp+0, -0x1.8c31a8ddc0000p-4},
    {0x1.187fe81914b87p+0, -0x1.765a9532e0000p-4}, {0x1.1780271da1a98p+0, -0x1.67bd4461f0000p-4},
    {0x1.167ff35d3bba2p+0, -0x1.590bf6081c000p-4}, {0x1.15001c50506c3p+0, -0x1.42ef6e9728000p-4},
    {0x1.13ffbd5e9c32cp+0, -0x1.34199c8bb8000p-4}, {0x1.12ffcf52edd20p+0, -0x1.253c8dee64000p-4},
    {0x1.118039be4b953p+0, -0x1.0edb9a7c14000p-4}, {0x1.107ff83cb5bf7p+0, -0x1.ffada7bb08000p-5},
    {0x1.0f7fd884cfae9p+0, -0x1.e18bc97cc8000p-5}, {0x1.0e001413eb252p+0, -0x1.b430383e70000p-5},
    {0x1.0cffd6b6ebd99p+0, -0x1.95c347a268000p-5}, {0x1.0bffcf347c818p+0, -0x1.773fbbdc80000p-5},
    {0x1.0b0016d6fa7fcp+0, -0x1.58a877bf60000p-5}, {0x1.0a000cbb82e82p+0, -0x1.39ea03bf08000p-5},
    {0x1.090037fe01c38p+0, -0x1.1b145b77a8000p-5}, {0x1.077ffe18877a6p+0, -0x1.d919f05f20000p-6},
    {0x1.068036d8c169dp+0, -0x1.9adbd49580000p-6}, {0x1.05802a65880edp+0, -0x1.5c50056b00000p-6},
    {0x1.047fccfab3a8dp+0, -0x1.1d72f5cdc0000p-6}, {0x1.037fc558de5bcp+0, -0x1.bcda247540000p-7},
    {0x1.027fc3984b664p+0, -0x1.3e54acbb40000p-7}, {1.0, 0.0},
    {1.0, 0.0}, {1.0, 0.0},
    {0x1.f9ff864c573ffp-1, 0x1.8263538240000p-7}, {0x1.f5ffebc30659bp-1, 0x1.432d26df60000p-6},
    {0x1.f2000fe6bf4b2p-1, 0x1.c63b239b60000p-6}, {0x1.eeffb8e05215ap-1, 0x1.14a2d75040000p-5},
    {0x1.eb00752bcbe80p-1, 0x1.570e21d5c0000p-5}, {0x1.e7006bbf6bcd8p-1, 0x1.9a1166e180000p-5},
    {0x1.e3ffc9f832421p-1, 0x1.ccbacf5de8000p-5}, {0x1.e00066c3221cdp-1, 0x1.08561e72b8000p-4},
    {0x1.dcfff33a4d167p-1, 0x1.2208237470000p-4}, {0x1.d9004f435767bp-1, 0x1.448331daac000p-4},
    {0x1.d600604bceee9p-1, 0x1.5e925da3ec000p-4}, {0x1.d20012b70cfdap-1, 0x1.81973e742c000p-4},
    {0x1.cf0051acd1532p-1, 0x1.9c09604808000p-4}, {0x1.cc00567fcd61bp-1, 0x1.b6a986a300000p-4},
    {0x1.c90040e547d1fp-1, 0x1.d17732dcbc000p-4}, {0x1.c4ffc05e59bfbp-1, 0x1.f57e07333c000p-4},
    {0x1.c1ffdc55b2015p-1, 0x1.085a2daaf2000p-3}, {0x1.bf004695edbadp-1, 0x1.160b3cbe9c000p-3},
    {0x1.bbff98168df0dp-1, 0x1.23d8f1f2fe000p-3}, {0x1.b8ffc48feef5ap-1, 0x1.31baa8dafe000p-3},
    {0x1.b600252233021p-1, 0x1.3fb3acb886000p-3}, {0x1.b300541b46271p-1, 0x1.4dc62c9da8000p-3},
    {0x1.b0ffeff461d1ap-1, 0x1.5738187448000p-3}, {0x1.adffa7f4905aap-1, 0x1.65768f3f8a000p-3},
    {0x1.aaffa30c20200p-1, 0x1.73cd4e4836000p-3}, {0x1.a7ffb2d1b6c8cp-1, 0x1.823d8b217c000p-3},
    {0x1.a4ffc222ba90cp-1, 0x1.90c8089200000p-3}, {0x1.a2ffac38c7e32p-1, 0x1.9a89125d36000p-3},
    {0x1.a000480ab1191p-1, 0x1.a93d711e02000p-3}, {0x1.9cffe537e4d2ep-1, 0x1.b811f7d9d8000p-3},
    {0x1.9b004c3e5f5ebp-1, 0x1.c2010ec634000p-3}, {0x1.97ffb57b72f94p-1, 0x1.d104f53346000p-3},
    {0x1.96004732b4b08p-1, 0x1.db1273e7cc000p-3}, {0x1.93002b3504f33p-1, 0x1.ea436e5d80000p-3},
    {0x1.90ffd17c6e028p-1, 0x1.f4759ec3a6000p-3}, {0x1.8dffb32c1f74ap-1, 0x1.01ebab0d47000p-2},
    {0x1.8bffbe77b7280p-1, 0x1.07142f79fd000p-2}, {0x1.89ffc57fa3f9ap-1, 0x1.0c436e8176000p-2},
    {0x1.8700286941c88p-1, 0x1.1416151df7000p-2}, {0x1.84ffd1d4297c1p-1, 0x1.19574d4432000p-2},
    {0x1.83004a2a74548p-1, 0x1.1e9d523a8d000p-2}, {0x1.7fffc4d50f546p-1, 0x1.2696bedb31000p-2},
    {0x1.7dffa4a647851p-1, 0x1.2beffcae53000p-2}, {0x1.7bffc554137f1p-1, 0x1.314fbc3800000p-2},
    {0x1.79ffcdca39feap-1, 0x1.36b6ff70b8000p-2}, {0x1.77ffde1986d42p-1, 0x1.3c2583c635000p-2},
    {0x1.74ffabc4ffc28p-1, 0x1.445a05426a000p-2}, {0x1.72fff3a2dd6e2p-1, 0x1.49daa15bea000p-2},
    {0x1.710002fb688a1p-1, 0x1.4f63767527000p-2}, {0x1.6f0040944a349p-1, 0x1.54f37d8790000p-2},
    {0x1.6cffb4a754474p-1, 0x1.5a8d811dfc000p-2}, {0x1.6affc143d9873p-1, 0x1.602db9a7c3000p-2},
};

// ln x by a table-driven reduction (P. T. P. Tang, ACM Trans. Math. Softw. 16, 1990):
// x = 2^e m with m in [sqrt(1/2), sqrt(2)), z = m r - 1, |z| < 2^-7 (1.02),
//   ln x = e ln 2 - ln r + z + z^2 (-1/2 + z/3 - ... - z^6/8).
// ln 2 is split into its first 40 bits and the rest (W. J. Cody and W. Waite,
// Software Manual for the Elementary Functions, 1980), so that e times the first
// part, less ln r, is exact.  Within 0.76 ulp (CUDA's log: 1); a table of -ln r
// rounded to FP64 left 1.46.  log() for values that are not positive and normal
// (the test on the high word costs no FP64 instruction).
__device__ __forceinline__ double log64(double x) {
    const int hx = __double2hiint(x);
    if ((unsigned)(hx - 0x00100000) >= 0x7fe00000u) return log(x);
    const int i = hx - 0x3fe6a09e;
    const int e = i >> 20;
    const double m = __hiloint2double(hx - (e << 20), __double2loint(x));
    const double2 t = __ldg(&LOG64[(i >> 13) & 127]);
    const double ed = __hiloint2double(0x43300000, e ^ 0x80000000) - 4503601774854144.0;   // (double)e
    const double z = fma(m, t.x, -1.0);
    const double z2 = __dmul_rn(z, z);
    double p = fma(z, -1.0 / 8, 1.0 / 7);
    p = fma(z, p, -1.0 / 6);
    p = fma(z, p, 1.0 / 5);
    p = fma(z, p, -1.0 / 4);
    p = fma(z, p, 1.0 / 3);
    p = fma(z, p, -1.0 / 2);
    const double lo = fma(z2, p, __dmul_rn(ed, 0x1.9ef35793c7673p-41));
    const double hi = fma(ed, 0x1.62e42fefa2000p-1, t.y);
    return __dadd_rn(hi, __dadd_rn(z, lo));
}

// 1/x: the hardware's approximation r (2^-20) and one step of fourth order, r + r (h +
// h^2 + h^3), h = 1 - x r; what is left out, r h^4, is below 2^-80 of it, so that the
// one rounding at the end counts (within 0.501 ulp; without h^3 0.508).  For x and 1/x
// normal numbers: zero, infinities and numbers beyond give NaN (the kernels divide by
// 1/M_phi + K, Mbar, |grad phi|^2 + delta^2 and products of them, whose zeros and
// overflows make the rate NaN with IEEE divisions as well).
__device__ __forceinline__ double rcp64(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double h = fma(-x, r, 1.0);
    return fma(r, fma(h, fma(h, h, h), h), r);
}

}  // namespace pf

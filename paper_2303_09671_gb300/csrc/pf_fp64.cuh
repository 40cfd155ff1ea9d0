// pf_fp64.cuh -- FP64 logarithm and reciprocal for the step kernels, in fewer
// instructions of the FP64 pipe than log() and the IEEE division: a GB300's FP64
// pipe takes about 19 cycles per warp instruction and SM and bounds every FP64
// step.  The logarithm takes 14 of them, the reciprocal 3.
#pragma once
#include <cuda_runtime.h>

namespace pf {

// {r, -ln r}, r a ratio k/512 near the reciprocal of the centre of interval t of
// [sqrt(1/2), sqrt(2)) (128 intervals, equal in the bits of the double); r = 1 for
// the three intervals around 1, where the logarithm has to keep its relative error
static __device__ const double2 LOG64[128] = {
    {1.41015625, -0x1.5ff3070a793d4p-2}, {1.40234375, -0x1.5a42ab0f4cfe2p-2},
    {1.39453125, -0x1.548a2c3add263p-2}, {1.38671875, -0x1.4ec973260026ap-2},
    {1.380859375, -0x1.4a7373cecf997p-2}, {1.373046875, -0x1.44a41b463c47cp-2},
    {1.365234375, -0x1.3ecc460ef5f50p-2}, {1.357421875, -0x1.38ebdb38ed321p-2},
    {1.3515625, -0x1.347dd9a987d55p-2}, {1.34375, -0x1.2e8e2bae11d31p-2},
    {1.3359375, -0x1.2895a13de86a3p-2}, {1.330078125, -0x1.241558bfd1404p-2},
    {1.322265625, -0x1.1e0d0c33716bep-2}, {1.31640625, -0x1.1980d2dd4236fp-2},
    {1.30859375, -0x1.136870293a8b0p-2}, {1.302734375, -0x1.0ed005f657da4p-2},
    {1.296875, -0x1.0a324e27390e3p-2}, {1.2890625, -0x1.0402594b4d041p-2},
    {1.283203125, -0x1.feb0233e607ccp-3}, {1.27734375, -0x1.f550a564b7b37p-3},
    {1.26953125, -0x1.e8c0252aa5a60p-3}, {1.263671875, -0x1.df46c0c722d2fp-3},
    {1.2578125, -0x1.d5c216b4fbb91p-3}, {1.251953125, -0x1.cc320c0176502p-3},
    {1.24609375, -0x1.c2968558c18c1p-3}, {1.240234375, -0x1.b8ef670420c3bp-3},
    {1.234375, -0x1.af3c94e80bff3p-3}, {1.228515625, -0x1.a57df28244dcdp-3},
    {1.22265625, -0x1.9bb362e7dfb83p-3}, {1.216796875, -0x1.91dcc8c340bdep-3},
    {1.2109375, -0x1.87fa06520c911p-3}, {1.205078125, -0x1.7e0afd630c274p-3},
    {1.19921875, -0x1.740f8f54037a5p-3}, {1.193359375, -0x1.6a079d0f7aad2p-3},
    {1.1875, -0x1.5ff3070a793d4p-3}, {1.181640625, -0x1.55d1ad4232d6fp-3},
    {1.177734375, -0x1.4f099f4a230b2p-3}, {1.171875, -0x1.44d2b6ccb7d1ep-3},
    {1.166015625, -0x1.3a8eb2d31a376p-3}, {1.16015625, -0x1.303d718e47fd3p-3},
    {1.15625, -0x1.29552f81ff523p-3}, {1.150390625, -0x1.1eed90e2dc2c3p-3},
    {1.14453125, -0x1.14785846742acp-3}, {1.140625, -0x1.0d77e7cd08e59p-3},
    {1.134765625, -0x1.02ebb42bf3d4bp-3}, {1.130859375, -0x1.f7b79fec37ddfp-4},
    {1.125, -0x1.e27076e2af2e6p-4}, {1.12109375, -0x1.d4313d66cb35dp-4},
    {1.115234375, -0x1.beba818146765p-4}, {1.111328125, -0x1.b05b49bee43fep-4},
    {1.10546875, -0x1.9ab42462033adp-4}, {1.1015625, -0x1.8c345d6319b21p-4},
    {1.095703125, -0x1.765bf23a6be13p-4}, {1.091796875, -0x1.67bb0726ec0fcp-4},
    {1.087890625, -0x1.590cafdf01c28p-4}, {1.08203125, -0x1.42edcbea646f0p-4},
    {1.078125, -0x1.341d7961bd1d1p-4}, {1.07421875, -0x1.253f62f0a1417p-4},
    {1.068359375, -0x1.0ed839b5526fep-4}, {1.064453125, -0x1.ffae9119b9303p-5},
    {1.060546875, -0x1.e19070c276016p-5}, {1.0546875, -0x1.b42dd711971bfp-5},
    {1.05078125, -0x1.95c830ec8e3ebp-5}, {1.046875, -0x1.77458f632dcfcp-5},
    {1.04296875, -0x1.58a5bafc8e4d5p-5}, {1.0390625, -0x1.39e87b9febd60p-5},
    {1.03515625, -0x1.1b0d98923d980p-5}, {1.029296875, -0x1.d91a66c543cc4p-6},
    {1.025390625, -0x1.9ace7551cc514p-6}, {1.021484375, -0x1.5c45a51b8d389p-6},
    {1.017578125, -0x1.1d7f7eb9eebe7p-6}, {1.013671875, -0x1.bcf712c74384cp-7},
    {1.009765625, -0x1.3e7295d25a7d9p-7}, {1.0, 0x0.0p+0},
    {1.0, 0x0.0p+0}, {1.0, 0x0.0p+0},
    {0.98828125, 0x1.82448a388a2aap-7}, {0.98046875, 0x1.432a925980cc1p-6},
    {0.97265625, 0x1.c63d2ec14aaf2p-6}, {0.966796875, 0x1.149e3e4005a8dp-5},
    {0.958984375, 0x1.5715c4c03ceefp-5}, {0.951171875, 0x1.9a187b573de7cp-5},
    {0.9453125, 0x1.ccb73cdddb2ccp-5}, {0.9375, 0x1.08598b59e3a07p-4},
    {0.931640625, 0x1.2207b5c78549ep-4}, {0.923828125, 0x1.4485e03dbdfadp-4},
    {0.91796875, 0x1.5e95a4d9791cbp-4}, {0.91015625, 0x1.8197e2f40e3f0p-4},
    {0.904296875, 0x1.9c0c32d4d2548p-4}, {0.8984375, 0x1.b6ac88dad5b1cp-4},
    {0.892578125, 0x1.d179788219364p-4}, {0.884765625, 0x1.f57bc7d9005dbp-4},
    {0.87890625, 0x1.08598b59e3a07p-3}, {0.873046875, 0x1.160c8024b27b1p-3},
    {0.8671875, 0x1.23d712a49c202p-3}, {0.861328125, 0x1.31b994d3a4f85p-3},
    {0.85546875, 0x1.3fb45a59928ccp-3}, {0.849609375, 0x1.4dc7b897bc1c8p-3},
    {0.845703125, 0x1.5737cc9018cddp-3}, {0.83984375, 0x1.6574ebe8c133ap-3},
    {0.833984375, 0x1.73cb9074fd14dp-3}, {0.828125, 0x1.823c16551a3c2p-3},
    {0.822265625, 0x1.90c6db9fcbcd9p-3}, {0.818359375, 0x1.9a8778debaa38p-3},
    {0.8125, 0x1.a93ed3c8ad9e3p-3}, {0.806640625, 0x1.b811730b823d2p-3},
    {0.802734375, 0x1.c2028ab17f9b4p-3}, {0.796875, 0x1.d1037f2655e7bp-3},
    {0.79296875, 0x1.db13db0d48940p-3}, {0.787109375, 0x1.ea4449f04aaf5p-3},
    {0.783203125, 0x1.f474b134df229p-3}, {0.77734375, 0x1.01eae5626c691p-2},
    {0.7734375, 0x1.07138604d5862p-2}, {0.76953125, 0x1.0c42d676162e3p-2},
    {0.763671875, 0x1.14167ef367783p-2}, {0.759765625, 0x1.1956d3b9bc2fap-2},
    {0.755859375, 0x1.1e9e1678899f4p-2}, {0.75, 0x1.269621134db92p-2},
    {0.74609375, 0x1.2bef07cdc9354p-2}, {0.7421875, 0x1.314f1e1d35ce4p-2},
    {0.73828125, 0x1.36b6776be1117p-2}, {0.734375, 0x1.3c25277333184p-2},
    {0.728515625, 0x1.44591e0539f49p-2}, {0.724609375, 0x1.49da7f3bcc41fp-2},
    {0.720703125, 0x1.4f637ebba9810p-2}, {0.716796875, 0x1.54f431b7be1a9p-2},
    {0.712890625, 0x1.5a8cadbbedfa1p-2}, {0.708984375, 0x1.602d08af091ecp-2},
};

// ln x by a table-driven reduction (P. T. P. Tang, ACM Trans. Math. Softw. 16, 1990):
// x = 2^e m with m in [sqrt(1/2), sqrt(2)), z = m r - 1, |z| < 2^-7 (1.02),
//   ln x = e ln 2 - ln r + z + z^2 (-1/2 + z/3 - ... - z^6/8).
// Within about one ulp; log() for values that are not positive and normal (the
// test on the high word costs no FP64 instruction).
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
    const double hi = fma(ed, 0x1.62e42fefa2000p-1, t.y);   // the first 40 bits of ln 2: exact with e
    return __dadd_rn(hi, __dadd_rn(z, lo));
}

// 1/x within about one ulp: the hardware's approximation r (2^-23) and one step of
// third order, r + r (h + h^2), h = 1 - x r.
__device__ __forceinline__ double rcp64(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double h = fma(-x, r, 1.0);
    return fma(r, fma(h, h, h), r);
}

}  // namespace pf

// fp64_math.cuh -- short FP64 elementary functions for arguments that are known
// to be ordinary (finite, normal, not huge), where the general functions' cost
// matters: an FP64 warp instruction holds an SM's FP64 pipe for ~19 clocks, and
// the closed-form integrals of the near pairs and the FP64 quadrature are bound by the number of them.
//
//   rcp64, rsqrt64   the hardware seed (rcp/rsqrt.approx.ftz.f64, ~2^-20) and one Householder step of third order
//                    (error e^3): 3 and 5 FP64 operations
//   log64            table-driven (P. T. P. Tang, "Table-driven implementation of the logarithm function in IEEE
//                    floating-point arithmetic", ACM TOMS 16, 1990): x = 2^e m, m in [3/4, 3/2), r = m c - 1 with c
//                    near 1/m from 128 entries, log x = e ln 2 - log c + log1p(r), |r| <= 2^-7, by its series: 13
//   atan2_pos        angle of (d, n), n >= 0, in [0, pi]: t = min/max, c = the nearest k/64, atan t = atan c +
//                    atan((t - c)/(1 + t c)) by its series: ~20
//   sincos64         reduction by pi/2 in two FMAs, then the Taylor series on [-pi/4, pi/4]: 23
// Each is within about 2 units of the last place over the ranges used (tests/test_fp64_math_gpu.py).
#pragma once

#include <math.h>

namespace cbfm {
namespace f64 {

// {c, -log c}: c near the reciprocal of the centre of each of 64 intervals of [3/4, 1) and 64 of [1, 3/2); c = 1
// on both sides of 1, so that the logarithm keeps its relative accuracy there
static __device__ const double2 LOG_TAB[128] = {
    {0x1.5470000000000p+0, -0x1.23e5398b931d0p-2}, {0x1.52b0000000000p+0, -0x1.1e9e3678891f4p-2},
    {0x1.50f0000000000p+0, -0x1.195033b43fa99p-2}, {0x1.4f40000000000p+0, -0x1.142bfeb9a0474p-2},
    {0x1.4d80000000000p+0, -0x1.0ed005f657da4p-2}, {0x1.4bd0000000000p+0, -0x1.099e371c0bc82p-2},
    {0x1.4a20000000000p+0, -0x1.0465a08154ffap-2}, {0x1.4880000000000p+0, -0x1.feb0233e607ccp-3},
    {0x1.46e0000000000p+0, -0x1.f488311d1b493p-3}, {0x1.4540000000000p+0, -0x1.ea5349e23ac0ep-3},
    {0x1.43a0000000000p+0, -0x1.e0114c533197fp-3}, {0x1.4210000000000p+0, -0x1.d627d7c1b2da7p-3},
    {0x1.4080000000000p+0, -0x1.cc320c0176502p-3}, {0x1.3ef0000000000p+0, -0x1.c22fca31887ddp-3},
    {0x1.3d60000000000p+0, -0x1.b820f2fc7e508p-3}, {0x1.3bd0000000000p+0, -0x1.ae05669628825p-3},
    {0x1.3a50000000000p+0, -0x1.a4454820d19fap-3}, {0x1.38d0000000000p+0, -0x1.9a7938d209947p-3},
    {0x1.3750000000000p+0, -0x1.90a11b46b9b56p-3}, {0x1.35e0000000000p+0, -0x1.8726935acac62p-3},
    {0x1.3460000000000p+0, -0x1.7d36832b8f0e3p-3}, {0x1.32f0000000000p+0, -0x1.73a4d01722e5cp-3},
    {0x1.3180000000000p+0, -0x1.6a079d0f7aad2p-3}, {0x1.3020000000000p+0, -0x1.60ca8fe8858afp-3},
    {0x1.2eb0000000000p+0, -0x1.57168c4aff0e6p-3}, {0x1.2d50000000000p+0, -0x1.4dc378969b1c1p-3},
    {0x1.2bf0000000000p+0, -0x1.446579dc223dep-3}, {0x1.2a90000000000p+0, -0x1.3afc766c1e210p-3},
    {0x1.2930000000000p+0, -0x1.3188543c098a1p-3}, {0x1.27e0000000000p+0, -0x1.2877bbc0b6ba6p-3},
    {0x1.2690000000000p+0, -0x1.1f5cd21a0d938p-3}, {0x1.2540000000000p+0, -0x1.16377fb124192p-3},
    {0x1.23f0000000000p+0, -0x1.0d07ac9dcbcf8p-3}, {0x1.22a0000000000p+0, -0x1.03cd40a51ac0dp-3},
    {0x1.2150000000000p+0, -0x1.f510466fd80bfp-4}, {0x1.2010000000000p+0, -0x1.e353fec9a2699p-4},
    {0x1.1ed0000000000p+0, -0x1.d183f87ea737cp-4}, {0x1.1d90000000000p+0, -0x1.bfa007672aa23p-4},
    {0x1.1c50000000000p+0, -0x1.ada7fec6ac801p-4}, {0x1.1b10000000000p+0, -0x1.9b9bb14949167p-4},
    {0x1.19e0000000000p+0, -0x1.8a6377a915c29p-4}, {0x1.18b0000000000p+0, -0x1.7918a1bf981d6p-4},
    {0x1.1780000000000p+0, -0x1.67bb0726ec0fcp-4}, {0x1.1650000000000p+0, -0x1.564a7ef514311p-4},
    {0x1.1520000000000p+0, -0x1.44c6dfb9b7606p-4}, {0x1.13f0000000000p+0, -0x1.332fff7bd1f18p-4},
    {0x1.12d0000000000p+0, -0x1.22743457a9c8ep-4}, {0x1.11a0000000000p+0, -0x1.10b75afd660c6p-4},
    {0x1.1080000000000p+0, -0x1.ffae9119b9303p-5}, {0x1.0f60000000000p+0, -0x1.ddcaadb46ef1bp-5},
    {0x1.0e40000000000p+0, -0x1.bbc2bfc44f417p-5}, {0x1.0d20000000000p+0, -0x1.99967a4f2b1c8p-5},
    {0x1.0c10000000000p+0, -0x1.792e93e5199edp-5}, {0x1.0af0000000000p+0, -0x1.56bac43ed7f9ap-5},
    {0x1.09e0000000000p+0, -0x1.360ebf5d83765p-5}, {0x1.08d0000000000p+0, -0x1.15413ca0e72a8p-5},
    {0x1.07c0000000000p+0, -0x1.e8a3ee30cdcacp-6}, {0x1.06b0000000000p+0, -0x1.a68151fb5c04ap-6},
    {0x1.05a0000000000p+0, -0x1.641a176270d6fp-6}, {0x1.0490000000000p+0, -0x1.216daf6d9321ap-6},
    {0x1.0390000000000p+0, -0x1.c4db352e6d472p-7}, {0x1.0280000000000p+0, -0x1.3e7295d25a7d9p-7},
    {0x1.0180000000000p+0, -0x1.7ee11ebd82e94p-8}, {0x1.0000000000000p+0, 0x0.0p+0},
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.fa20000000000p-1, 0x1.7a2c82e212c65p-7},
    {0x1.f640000000000p-1, 0x1.3b024b78c5669p-6}, {0x1.f260000000000p-1, 0x1.b9e8027e1918ep-6},
    {0x1.eea0000000000p-1, 0x1.1ad398c6cd588p-5}, {0x1.eae0000000000p-1, 0x1.592bbc15215c9p-5},
    {0x1.e740000000000p-1, 0x1.95e430f8ce45ep-5}, {0x1.e3a0000000000p-1, 0x1.d310ba20455a1p-5},
    {0x1.e020000000000p-1, 0x1.074883629640bp-4}, {0x1.dca0000000000p-1, 0x1.254062f0a9417p-4},
    {0x1.d920000000000p-1, 0x1.4370ce02b7de8p-4}, {0x1.d5c0000000000p-1, 0x1.60c38ba79945dp-4},
    {0x1.d280000000000p-1, 0x1.7d33687c293c9p-4}, {0x1.cf20000000000p-1, 0x1.9af124d64c626p-4},
    {0x1.cbe0000000000p-1, 0x1.b7c9832f5801ap-4}, {0x1.c8c0000000000p-1, 0x1.d3b73f37e1f9bp-4},
    {0x1.c580000000000p-1, 0x1.f0f70cdd992e3p-4}, {0x1.c260000000000p-1, 0x1.06a4d1d26c5e6p-3},
    {0x1.bf60000000000p-1, 0x1.1454d8953741cp-3}, {0x1.bc40000000000p-1, 0x1.22aff2ddbd971p-3},
    {0x1.b960000000000p-1, 0x1.2ffbf29a6645cp-3}, {0x1.b660000000000p-1, 0x1.3df3ab13505f7p-3},
    {0x1.b380000000000p-1, 0x1.4b6d6fefe22a4p-3}, {0x1.b0a0000000000p-1, 0x1.58fe0e4c62eaep-3},
    {0x1.adc0000000000p-1, 0x1.66a5d42a3ad34p-3}, {0x1.ab00000000000p-1, 0x1.73cb9074fd14dp-3},
    {0x1.a820000000000p-1, 0x1.81a18b4220535p-3}, {0x1.a580000000000p-1, 0x1.8e588ebac2dbfp-3},
    {0x1.a2c0000000000p-1, 0x1.9bc062f26fc3ap-3}, {0x1.a020000000000p-1, 0x1.a8a14ffee66bdp-3},
    {0x1.9d80000000000p-1, 0x1.b5971a213acdbp-3}, {0x1.9ae0000000000p-1, 0x1.c2a205610593fp-3},
    {0x1.9860000000000p-1, 0x1.cf21d5ecbaa65p-3}, {0x1.95c0000000000p-1, 0x1.dc56cae452f5ap-3},
    {0x1.9340000000000p-1, 0x1.e8ff2622babc7p-3}, {0x1.90e0000000000p-1, 0x1.f518262c38082p-3},
    {0x1.8e60000000000p-1, 0x1.00f40470c7324p-2}, {0x1.8c00000000000p-1, 0x1.07138604d5862p-2},
    {0x1.89a0000000000p-1, 0x1.0d3c7586cd5e4p-2}, {0x1.8740000000000p-1, 0x1.136ef02e8290cp-2},
    {0x1.8500000000000p-1, 0x1.1956d3b9bc2fap-2}, {0x1.82a0000000000p-1, 0x1.1f9c39f74c557p-2},
    {0x1.8060000000000p-1, 0x1.2596410df963ap-2}, {0x1.7e20000000000p-1, 0x1.2b9943b06bd76p-2},
    {0x1.7be0000000000p-1, 0x1.31a55d07a8591p-2}, {0x1.79c0000000000p-1, 0x1.3763e64645463p-2},
    {0x1.77a0000000000p-1, 0x1.3d2abb3b3b4dfp-2}, {0x1.7560000000000p-1, 0x1.4351b33743eb9p-2},
    {0x1.7340000000000p-1, 0x1.4929e8db4e6e4p-2}, {0x1.7140000000000p-1, 0x1.4eb1f36b07184p-2},
    {0x1.6f20000000000p-1, 0x1.549aec5def881p-2}, {0x1.6d20000000000p-1, 0x1.5a32eb2e4eacbp-2},
    {0x1.6b20000000000p-1, 0x1.5fd2c78c78828p-2}, {0x1.6920000000000p-1, 0x1.657a97b64d437p-2},
    {0x1.6720000000000p-1, 0x1.6b2a72488ad8fp-2}, {0x1.6520000000000p-1, 0x1.70e26e40eb5fap-2},
    {0x1.6340000000000p-1, 0x1.76466197e36dep-2}, {0x1.6140000000000p-1, 0x1.7c0e612785c73p-2},
    {0x1.5f60000000000p-1, 0x1.81818203afc80p-2}, {0x1.5d80000000000p-1, 0x1.86fc19d05148ep-2},
    {0x1.5ba0000000000p-1, 0x1.8c7e3d1c80b30p-2}, {0x1.59e0000000000p-1, 0x1.91a93f1f4a7a8p-2},
    {0x1.5800000000000p-1, 0x1.973a3431356aep-2}, {0x1.5640000000000p-1, 0x1.9c73305d47ebbp-2}};
// {k / 64, atan(k / 64)}
static __device__ const double2 ATAN_TAB[65] = {
    {0x0.0p+0, 0x0.0p+0}, {0x1.0000000000000p-6, 0x1.fff555bbb729bp-7},
    {0x1.0000000000000p-5, 0x1.ffd55bba97625p-6}, {0x1.8000000000000p-5, 0x1.7fb818430da2ap-5},
    {0x1.0000000000000p-4, 0x1.ff55bb72cfdeap-5}, {0x1.4000000000000p-4, 0x1.3f59f0e7c559dp-4},
    {0x1.8000000000000p-4, 0x1.7ee182602f10fp-4}, {0x1.c000000000000p-4, 0x1.be39ebe6f07c3p-4},
    {0x1.0000000000000p-3, 0x1.fd5ba9aac2f6ep-4}, {0x1.2000000000000p-3, 0x1.1e1fafb043727p-3},
    {0x1.4000000000000p-3, 0x1.3d6eee8c6626cp-3}, {0x1.6000000000000p-3, 0x1.5c9811e3ec26ap-3},
    {0x1.8000000000000p-3, 0x1.7b97b4bce5b02p-3}, {0x1.a000000000000p-3, 0x1.9a6a8e96c8626p-3},
    {0x1.c000000000000p-3, 0x1.b90d7529260a2p-3}, {0x1.e000000000000p-3, 0x1.d77d5df205736p-3},
    {0x1.0000000000000p-2, 0x1.f5b75f92c80ddp-3}, {0x1.1000000000000p-2, 0x1.09dc597d86362p-2},
    {0x1.2000000000000p-2, 0x1.18bf5a30bf178p-2}, {0x1.3000000000000p-2, 0x1.278372057ef46p-2},
    {0x1.4000000000000p-2, 0x1.362773707ebccp-2}, {0x1.5000000000000p-2, 0x1.44aa436c2af0ap-2},
    {0x1.6000000000000p-2, 0x1.530ad9951cd4ap-2}, {0x1.7000000000000p-2, 0x1.614840309cfe2p-2},
    {0x1.8000000000000p-2, 0x1.6f61941e4def1p-2}, {0x1.9000000000000p-2, 0x1.7d5604b63b3f7p-2},
    {0x1.a000000000000p-2, 0x1.8b24d394a1b25p-2}, {0x1.b000000000000p-2, 0x1.98cd5454d6b18p-2},
    {0x1.c000000000000p-2, 0x1.a64eec3cc23fdp-2}, {0x1.d000000000000p-2, 0x1.b3a911da65c6cp-2},
    {0x1.e000000000000p-2, 0x1.c0db4c94ec9f0p-2}, {0x1.f000000000000p-2, 0x1.cde53432c1351p-2},
    {0x1.0000000000000p-1, 0x1.dac670561bb4fp-2}, {0x1.0800000000000p-1, 0x1.e77eb7f175a34p-2},
    {0x1.1000000000000p-1, 0x1.f40dd0b541418p-2}, {0x1.1800000000000p-1, 0x1.0039c73c1a40cp-1},
    {0x1.2000000000000p-1, 0x1.0657e94db30d0p-1}, {0x1.2800000000000p-1, 0x1.0c6145b5b43dap-1},
    {0x1.3000000000000p-1, 0x1.1255d9bfbd2a9p-1}, {0x1.3800000000000p-1, 0x1.1835a88be7c13p-1},
    {0x1.4000000000000p-1, 0x1.1e00babdefeb4p-1}, {0x1.4800000000000p-1, 0x1.23b71e2cc9e6ap-1},
    {0x1.5000000000000p-1, 0x1.2958e59308e31p-1}, {0x1.5800000000000p-1, 0x1.2ee628406cbcap-1},
    {0x1.6000000000000p-1, 0x1.345f01cce37bbp-1}, {0x1.6800000000000p-1, 0x1.39c391cd4171ap-1},
    {0x1.7000000000000p-1, 0x1.3f13fb89e96f4p-1}, {0x1.7800000000000p-1, 0x1.445065b795b56p-1},
    {0x1.8000000000000p-1, 0x1.4978fa3269ee1p-1}, {0x1.8800000000000p-1, 0x1.4e8de5bb6ec04p-1},
    {0x1.9000000000000p-1, 0x1.538f57b89061fp-1}, {0x1.9800000000000p-1, 0x1.587d81f732fbbp-1},
    {0x1.a000000000000p-1, 0x1.5d58987169b18p-1}, {0x1.a800000000000p-1, 0x1.6220d115d7b8ep-1},
    {0x1.b000000000000p-1, 0x1.66d663923e087p-1}, {0x1.b800000000000p-1, 0x1.6b798920b3d99p-1},
    {0x1.c000000000000p-1, 0x1.700a7c5784634p-1}, {0x1.c800000000000p-1, 0x1.748978fba8e0fp-1},
    {0x1.d000000000000p-1, 0x1.78f6bbd5d315ep-1}, {0x1.d800000000000p-1, 0x1.7d528289fa093p-1},
    {0x1.e000000000000p-1, 0x1.819d0b7158a4dp-1}, {0x1.e800000000000p-1, 0x1.85d69576cc2c5p-1},
    {0x1.f000000000000p-1, 0x1.89ff5ff57f1f8p-1}, {0x1.f800000000000p-1, 0x1.8e17aa99cc05ep-1},
    {0x1.0000000000000p+0, 0x1.921fb54442d18p-1}};

__device__ __forceinline__ double rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(fma(e, e, e), y, y);
}
__device__ __forceinline__ double rsqrt64(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double log64(double x) {
    const int hi = __double2hiint(x), d = hi - 0x3fe80000, e = d >> 20;
    const double m = __hiloint2double(hi - (e << 20), __double2loint(x));
    const double2 c = __ldg(&LOG_TAB[(d >> 13) & 127]);
    const double r = fma(m, c.x, -1.0);
    double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
    p = fma(r, p, -1.0 / 6.0);
    p = fma(r, p, 1.0 / 5.0);
    p = fma(r, p, -1.0 / 4.0);
    p = fma(r, p, 1.0 / 3.0);
    const double r2 = r * r;
    p = fma(r, p, -0.5);
    p = fma(r2, p, r);
    return fma((double)e, 0.69314718055994530942, c.y) + p;
}
__device__ __forceinline__ double atan2_pos(double n, double d) {
    const double PI_2 = 1.57079632679489661923;
    const double a = fabs(d);
    const bool swap = n > a;
    const double lo = swap ? a : n, hi = swap ? n : a;
    const int k = min(64, max(0, (int)fmaf((float)(lo * rcp64(hi)), 64.0f, 0.5f)));
    const double2 c = __ldg(&ATAN_TAB[k]);
    const double z = fma(-c.x, hi, lo) * rcp64(fma(c.x, lo, hi)), z2 = z * z;
    double p = fma(z2, -1.0 / 7.0, 1.0 / 5.0);
    p = fma(z2, p, -1.0 / 3.0);
    double t = c.y + fma(z * z2, p, z);
    if (swap) t = PI_2 - t;
    return d < 0.0 ? 2.0 * PI_2 - t : t;
}
__device__ __forceinline__ void sincos64(double x, double *s, double *c) {
    if (!(fabs(x) < 1e5)) {
        sincos(x, s, c);
        return;
    }
    const double SHIFT = 6755399441055744.0;   // 1.5 2^52
    const double t = fma(x, 0.63661977236758134308, SHIFT), n = t - SHIFT;
    const int q = __double2loint(t);
    double r = fma(n, -1.57079632679489655800, x);        // double(pi / 2): the product is exact in the FMA
    r = fma(n, -6.12323399573676603587e-17, r);           // pi / 2 - double(pi / 2)
    const double r2 = r * r;
    double a = fma(r2, -1.0 / 1307674368000.0, 1.0 / 6227020800.0);
    a = fma(r2, a, -1.0 / 39916800.0);
    a = fma(r2, a, 1.0 / 362880.0);
    a = fma(r2, a, -1.0 / 5040.0);
    a = fma(r2, a, 1.0 / 120.0);
    a = fma(r2, a, -1.0 / 6.0);
    a = fma(r2 * r, a, r);
    double b = fma(r2, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
    b = fma(r2, b, 1.0 / 479001600.0);
    b = fma(r2, b, -1.0 / 3628800.0);
    b = fma(r2, b, 1.0 / 40320.0);
    b = fma(r2, b, -1.0 / 720.0);
    b = fma(r2, b, 1.0 / 24.0);
    b = fma(r2, b, -0.5);
    b = fma(r2, b, 1.0);
    const double sv = (q & 1) ? b : a, cv = (q & 1) ? a : b;
    *s = (q & 2) ? -sv : sv;
    *c = ((q + 1) & 2) ? -cv : cv;
}

}  // namespace f64
}  // namespace cbfm

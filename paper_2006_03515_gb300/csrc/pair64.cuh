// The paper's kernel K(R) = (e^{-aR} - e^{-bR}) / (4 pi R^3 ln(b/a)) in FP64 from a squared distance,
// for the pair loops.
//
// What bounds those loops is the FP64 pipe: a GB300 SM has two FP64 lanes, a warp instruction takes 16
// cycles, and the pair written with sqrt, exp, expm1 and a division took about 75 of them (k_p2p,
// 48^3 points: 10.4 ms). Here it takes 38 (6.4 ms; k_p2m 2.09 -> 1.25 ms, k_l2p 2.44 -> 1.47 ms):
//  * 1/R: the hardware's approximate reciprocal square root and one third-order step,
//    y (1 + e/2 + 3 e^2/8) with e = 1 - r2 y^2 (the binomial series; the next term is 5 e^3/16, below
//    1e-17 for e < 3e-6);
//  * the exponentials by Tang's table-driven method (ACM TOMS 15, 1989): 2^t with t = k/256 + f/256,
//    |f| <= 1/2, from 256 tabulated powers and the Taylor polynomial of 2^{f/256} - 1;
//  * e^{-aR} - e^{-bR} = e^{-aR} (1 - e^{-(b-a)R}), the bracket from a second table of 1 - 2^{-j/256},
//    so that it keeps its relative precision where (b-a)R is small (degree 5 there, since the
//    polynomial then is the result).
// A block builds the tables in shared memory (one entry of each per thread of 256) with CUDA's own
// exp2 and expm1, or copies them from the plan. The FMM's results moved by 3e-16.
#pragma once
#include <cmath>

#include "kernel.cuh"

namespace kifmm {

constexpr int kPairTab = 256;   // table entries per octave

struct Pair64Tab {
    double t[kPairTab];   // 2^{-j/256}
    double m[kPairTab];   // 1 - 2^{-j/256}
};

// by all threads of the block; the caller synchronises
__device__ __forceinline__ void pair64_tab_fill(Pair64Tab& tab) {
    for (int j = threadIdx.x; j < kPairTab; j += blockDim.x) {
        tab.t[j] = exp2(-(double)j / kPairTab);
        tab.m[j] = -expm1(-(double)j * (0.69314718055994530942 / kPairTab));
    }
}

struct Pair64 {
    double ca, cm;       // a, b - a in units of ln2 / 256 per cm, and what their rounding left
    double cal, cml;     // (without it e^{-aR} is off by aR ulps for every pair alike)
    double ra, rm;       // R beyond which e^{-aR}, e^{-(b-a)R} are taken at the bound (below 1e-300)
    double norm;
};

inline Pair64 make_pair64(const KParams& k) {
    const double c = kPairTab * 1.4426950408889634074, cl = kPairTab * 2.0355273740931033e-17;   // 256 log2(e)
    const double ca = k.a * c, cm = k.bma * c;
    return Pair64{ca, cm, fma(k.a, c, -ca) + k.a * cl, fma(k.bma, c, -cm) + k.bma * cl, 690.0 / k.a, 690.0 / k.bma,
                  k.norm};
}

// x with min(x, hi) for x >= 0 by integer comparison of the high words (within 1e-6 of hi); NaN stays
__device__ __forceinline__ double pair64_min(double x, double hi) {
    const int xh = __double2hiint(x), hh = __double2hiint(hi);
    return xh > hh && xh < 0x7ff00000 ? hi : x;
}

// 1 / sqrt(x), x > 0: the approximate reciprocal square root and one third-order step
__device__ __forceinline__ double rsqrt64(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// e^{-x} for x >= 0 (0 above 690)
__device__ __forceinline__ double exp_neg64(double x, const Pair64Tab& tab) {
    constexpr double L = 0.69314718055994530942 / kPairTab, MAGIC = 6755399441055744.0;
    constexpr double c = kPairTab * 1.4426950408889634074, cl = kPairTab * 2.0355273740931033e-17;
    const double X = pair64_min(x, 691.0);
    double k = fma(X, c, MAGIC);
    const int i = __double2loint(k);
    k -= MAGIC;
    const double f = fma(-X, cl, fma(-X, c, k));
    double p = fma(f, L * L * L * L / 24, L * L * L / 6);
    p = fma(p, f, L * L / 2);
    p = fma(p, f, L);
    p *= f;
    double s = tab.t[i & (kPairTab - 1)];
    s = __hiloint2double(__double2hiint(s) - ((i >> 8) << 20), __double2loint(s));
    return __double2hiint(X) > __double2hiint(690.0) ? 0.0 : fma(s, p, s);
}

// e^{-aR} - e^{-bR} times norm / R^3; r2 > 0, 0 for an infinite r2 (taken as 2^996)
__device__ __forceinline__ double pair64_kernel(double r2, const Pair64& k, const Pair64Tab& tab) {
    constexpr double L = 0.69314718055994530942 / kPairTab;   // ln2 / 256
    constexpr double MAGIC = 6755399441055744.0;              // 1.5 2^52: x + MAGIC holds rint(x) in its low word
    const int r2h = __double2hiint(r2);
    r2 = __hiloint2double(r2h == 0x7ff00000 ? 0x7e300000 : r2h, __double2loint(r2));
    const double y = rsqrt64(r2);
    const double R = r2 * y;
    // e^{-aR} = s (1 + p): s = 2^{-ka/256}
    const double Ra = pair64_min(R, k.ra), Rm = pair64_min(R, k.rm);
    double ka = fma(Ra, k.ca, MAGIC);
    const int ia = __double2loint(ka);
    ka -= MAGIC;
    double f = fma(-Ra, k.cal, fma(-Ra, k.ca, ka));   // (256 log2 of the rest, |f| <= 1/2)
    double p = fma(f, L * L * L * L / 24, L * L * L / 6);
    p = fma(p, f, L * L / 2);
    p = fma(p, f, L);
    p *= f;
    double s = tab.t[ia & (kPairTab - 1)];
    s = __hiloint2double(__double2hiint(s) - ((ia >> 8) << 20), __double2loint(s));
    const double ea = fma(s, p, s);
    // 1 - e^{-(b-a)R} = (1 - s) - s p
    double km = fma(Rm, k.cm, MAGIC);
    const int im = __double2loint(km);
    km -= MAGIC;
    f = fma(-Rm, k.cml, fma(-Rm, k.cm, km));
    p = fma(f, L * L * L * L * L / 120, L * L * L * L / 24);
    p = fma(p, f, L * L * L / 6);
    p = fma(p, f, L * L / 2);
    p = fma(p, f, L);
    p *= f;
    s = tab.t[im & (kPairTab - 1)];
    s = __hiloint2double(__double2hiint(s) - ((im >> 8) << 20), __double2loint(s));
    const double om = (im >> 8) == 0 ? tab.m[im & (kPairTab - 1)] : 1.0 - s;
    const double bm = fma(-s, p, om);
    return (ea * bm) * (y * y) * (y * k.norm);
}

}  // namespace kifmm

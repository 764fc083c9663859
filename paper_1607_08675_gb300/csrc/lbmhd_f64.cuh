// lbmhd_f64.cuh -- the FP64 collision of one node, stored populations to
// stored populations, for the one-step kernels.
//
// The FP64 step is bound by the FP64 pipe (about 2 operations per SM and
// clock), so this form counts operations: 119 and three reciprocals and three
// square roots of 3 and 6 operations, 146 in all, against 216 of collide().
//  - Populations are not decoded and encoded: the differences of opposite
//    ones need no weight, a sum takes its weight in its first subtraction
//    (f - 2 w is exact near w, as f - w is), and the change is subtracted from
//    the population itself -- one rounding less.
//  - n5 = 2 (d5 - d6 + d8 - d7) - (d1 - d3) and n6 alike; quadratic terms are
//    accumulated onto their moments; constants are folded into the rates.
//  - Reciprocal and square root start from FP32 ones, whose operands and
//    results move between the formats by integer operations.  The reciprocal
//    takes one step of third order, y0 (1 + e + e^2); the root one of
//    Goldschmidt's steps and a correction by its exact remainder (Markstein).
//    Both are within 0.501 units of the last place (e is at most 2^-22), so
//    they differ from the IEEE ones in an occasional last place.  Operands
//    outside the range of the FP32 start, 2^-120 to 2^120, take the IEEE ones.
// Every operation is rounded as written, so all kernels give the same bits.
// ncu, 2048^2, one node per thread: the FP64 pipe 86% busy, issue 10%, DRAM 13%.
// Measured (GB300, us per step, collide() / this, one node per thread):
// 1024^2 399.5 / 295.4, 256^2 28.7 / 21.6, 64^2 8.5 / 6.6.
#pragma once

#include "lbmhd_device.cuh"

namespace lbmhd {

__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }

// The leading 24 bits of x as FP32, for 2^-120 <= |x| < 2^120.
__device__ __forceinline__ float cut_f64(double x) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    return __uint_as_float((h & 0x80000000u) | (((h & 0x7fffffffu) - (896u << 20)) << 3 | l >> 29));
}
__device__ __forceinline__ bool in_f32_range(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) - (903u << 20) < (240u << 20);
}
// A normal FP32 value, widened and scaled by 2^k.
__device__ __forceinline__ double put_f64(float v, int k = 0) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((896u + (unsigned)k) << 20))),
                            (int)(b << 29));
}

// 1 / x: y0 (1 + e + e^2), e = 1 - x y0, |e| <= 2^-22.
__device__ __forceinline__ double rcp64(double x) {
    if (!in_f32_range(x)) return 1.0 / x;
    const double y0 = put_f64(rcp(cut_f64(x)));
    const double e = fma_(-x, y0, 1.0);
    return fma_(y0, fma_(e, e, e), y0);
}
__device__ __forceinline__ double sqrt64(double x) {
    if (!in_f32_range(x) || __double2hiint(x) < 0) return sqrt(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(cut_f64(x)));
    const double h0 = put_f64(y, -1);      // 1 / (2 sqrt x)
    const double g0 = mul_(x, put_f64(y));  // sqrt x
    const double r = fma_(-g0, h0, 0.5);
    const double g1 = fma_(g0, r, g0), h1 = fma_(h0, r, h0);
    return fma_(fma_(-g1, g1, x), h1, g1);
}

// f[9], g[10]: the streamed populations, overwritten by the relaxed ones.
// See collide() for the moments, rates and equilibria.
__device__ __forceinline__ void collide64(double (&f)[9], double (&g)[10], const Coll<double>& c) {
    constexpr double w0 = 4.0 / 9.0, w1 = 1.0 / 9.0, w5 = 1.0 / 36.0;
    constexpr double k1_3 = 1.0 / 3.0, k1_6 = 1.0 / 6.0, k5_3 = 5.0 / 3.0;
    const double e13 = sub_(f[1], f[3]), e24 = sub_(f[2], f[4]), e56 = sub_(f[5], f[6]), e87 = sub_(f[8], f[7]);
    const double s13 = add_(sub_(f[1], 2.0 * w1), f[3]), s24 = add_(sub_(f[2], 2.0 * w1), f[4]);
    const double s56 = add_(sub_(f[5], 2.0 * w5), f[6]), s78 = add_(sub_(f[7], 2.0 * w5), f[8]);
    const double d0 = sub_(f[0], w0), dsum = add_(s56, s78), d0s = add_(d0, dsum), rt = add_(s13, s24);
    const double dsum9 = add_(d0s, rt);
    const double irho = rcp64(add_(1.0, dsum9));
    const double ab = add_(e56, e87), ce = sub_(s56, s78);
    const double jx = add_(e13, ab), jy = add_(e24, ce);
    const double ux = mul_(jx, irho), uy = mul_(jy, irho);
    const double bx = add_(add_(add_(g[0], g[2]), add_(g[4], g[6])), g[8]);
    const double by = add_(add_(add_(g[1], g[3]), add_(g[5], g[7])), g[9]);
    const double j2i = fma_(jx, ux, mul_(jy, uy));
    const double n3 = fma_(bx, by, fma_(-jx, uy, sub_(e56, e87)));
    const double n4 = fma_(-by, by, fma_(bx, bx, fma_(jy, uy, fma_(-jx, ux, sub_(s13, s24)))));
    const double n5 = fma_(2.0, ab, -e13), n6 = fma_(2.0, ce, -e24);
    const double n7q = fma_(0.75, j2i, fma_(-1.25, rt, d0s));  // n7 / 4
    const double n8 = fma_(3.0, j2i, fma_(-k5_3, dsum9, fma_(4.0, d0, -dsum)));
    const double E = fma_(ux, by, -mul_(uy, bx));

    double t2 = add_(c.tn, c.tn), m2 = add_(c.te, c.te);  // 2 tau_e, 2 tau_m
    if (c.les) {
        const double Q = sqrt64(fma_(n4, n4, mul_(4.0, mul_(n3, n3))));
        t2 = add_(c.tn, sqrt64(fma_(mul_(c.k18, Q), irho, c.tn2)));
        const double J = fabs(fma_(-2.0, E, sub_(sub_(g[3], g[7]), sub_(g[4], g[8]))));
        m2 = add_(c.te, sqrt64(fma_(c.k36, J, c.te2)));
    }
    const double rn = rcp64(t2), rm = rcp64(m2);  // s_nu / 2, s_m / 2
    const double hr = mul_(0.5, rn);
    const double a3 = mul_(hr, n3), a4 = mul_(hr, n4);
    const double a5 = mul_(c.c5, n5), a6 = mul_(c.c6, n6);
    const double a7 = mul_(c.fix7 ? c.c7 : mul_(rn, 2.0 / 45.0), n7q);
    const double a8 = mul_(c.fix8 ? c.c8 : mul_(rn, 0.1), n8);
    const double q78 = fma_(4.0, a7, -a8);
    const double u13 = fma_(-5.0, a7, a4), u24 = fma_(5.0, a7, a4);
    f[0] = fma_(-4.0, add_(a7, a8), f[0]);
    f[1] = sub_(f[1], fma_(-2.0, a5, u13));
    f[2] = add_(f[2], fma_(2.0, a6, u24));
    f[3] = sub_(f[3], fma_(2.0, a5, u13));
    f[4] = add_(f[4], fma_(-2.0, a6, u24));
    const double P = add_(a3, a5), M = sub_(a3, a5), S = add_(a6, q78), D = sub_(q78, a6);
    f[5] = sub_(f[5], add_(P, S));
    f[6] = sub_(f[6], sub_(S, P));
    f[7] = sub_(f[7], add_(M, D));
    f[8] = sub_(f[8], sub_(D, M));

    const double nsm = mul_(-2.0, rm);
    const double yp = fma_(3.0, E, by), ym = fma_(-3.0, E, by), xp = fma_(3.0, E, bx), xm = fma_(-3.0, E, bx);
    auto relax = [&](int q, double k, double v) { g[q] = fma_(nsm, fma_(-k, v, g[q]), g[q]); };
    relax(0, k1_3, bx);
    relax(1, k1_3, by);
    relax(2, k1_6, bx);
    relax(3, k1_6, yp);
    relax(4, k1_6, xm);
    relax(5, k1_6, by);
    relax(6, k1_6, bx);
    relax(7, k1_6, ym);
    relax(8, k1_6, xp);
    relax(9, k1_6, by);
}

}  // namespace lbmhd

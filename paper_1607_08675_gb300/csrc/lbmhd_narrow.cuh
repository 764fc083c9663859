// lbmhd_narrow.cuh -- FP64 in and out of the FP32 forms without the FP64 pipe.
//
// GB300 issues about 2 FP64 operations (conversions included) per SM and
// clock against 128 FP32 ones.  Initialisation takes FP64 fields to FP32
// populations and read-back takes FP32 populations to FP64 fields; both were
// bound by that rate, 8 to 14 times their memory time.
//
// Initialisation: the equilibria are formed in double-word FP32
// (lbmhd_ff.cuh) with a bound on their error, and rounded to FP32.  Where
// the bound leaves the rounding open the node takes the FP64 path, so the
// stored values are those of FP64 arithmetic whatever the input (a zero may
// lose its sign).
//
// Measured on GB300 (ms, before -> after): init of 8192^2 FP16 18.55 -> 3.44,
// 1999 x 1201 FP32 deviations 0.593 -> 0.115, 256^3 FP32 13.34 -> 2.53 (FP32
// issue now); moments of 8192^2 FP16 8.65 -> 4.86, 256^3 FP32 6.56 -> 2.39
// (still the FP64 rate, at less than half the operations).
#pragma once

#include <cuda_fp16.h>

#include "lbmhd_ff.cuh"

namespace lbmhd {

// x to 2^-49 of itself, in integer operations.  Zero, or 2^-60 <= |x| < 2^60;
// anything else clears ok.
__device__ __forceinline__ ff split_f64(double x, bool& ok) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const int e = (int)(h >> 20 & 0x7ffu) - 1023;
    const bool zero = ((h & 0x7fffffffu) | l) == 0u;
    ok = ok && (zero || (e >= -60 && e < 60));
    const unsigned sign = h & 0x80000000u;
    // the leading 23 fraction bits, then the other 29 as an integer
    const float hi = __uint_as_float(sign | (unsigned)(e + 127) << 23 | (h & 0xfffffu) << 3 | l >> 29);
    const float lo = __fmul_rn(__uint2float_rn(l & 0x1fffffffu),
                               __uint_as_float(sign | (unsigned)(e - 52 + 127) << 23));
    const ff r = fast_two_sum(hi, lo);
    return zero ? ff(0.0f, 0.0f) : r;
}

// FP32 rounding of a value known to within err of x.  open: a rounding
// boundary lies that near (or x is not a normal number).  Half the spacing
// at hi is 2^-24 of its power of two; below a power of two it is half that,
// which stands for both sides there.
__device__ __forceinline__ float round_ff(ff x, float err, bool& open) {
    const unsigned b = __float_as_uint(x.hi);
    float half_ulp = __uint_as_float((b & 0x7f800000u) - (24u << 23));
    if ((b & 0x7fffffu) == 0u) half_ulp *= 0.5f;
    const bool fine = (b & 0x7f800000u) >= (40u << 23) && (b & 0x7f800000u) < (200u << 23) &&
                      fabsf(x.lo) + err < half_ulp;
    // an exact zero: no term of the sum was there
    open = open || !(fine || (x.hi == 0.0f && err == 0.0f));
    return x.hi;
}

// The same for a value that is stored in binary16: an open FP32 rounding
// matters only where both FP32 neighbours do not round to one half.
__device__ __forceinline__ unsigned short round_ff_half(ff x, float err, bool& open) {
    bool o = false;
    const float f = round_ff(x, err, o);
    const unsigned short h = __half_as_ushort(__float2half_rn(f));
    if (o) {
        const float d = err + fabsf(f) * 0x1p-22f;
        const unsigned short p = __half_as_ushort(__float2half_rn(f - d)),
                             q = __half_as_ushort(__float2half_rn(f + d));
        open = open || !(p == q && h == p && fabsf(f) < 1e30f);
    }
    return h;
}

// An FP32 value as FP64 by moving its bits.  Denormals, infinities and NaN
// set odd (their bits mean something else).
__device__ __forceinline__ double widen_f32(float v, bool& odd) {
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    odd = odd || (m - 1u < 0x7fffffu) || m >= 0x7f800000u;
    const unsigned h = m ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)((b & 0x80000000u) | h), (int)(b << 29));
}

// n[i] / d for i < N (finite n) with one reciprocal: FP32 seed, one step of
// third order in FP64, and the quotient corrected by its exact remainder
// (Markstein), two multiply-adds after the product.  Within 0.501 units of the
// last place, so the IEEE quotient but for an occasional last place (a zero may
// lose its sign); divisors beyond 2^-60 to 2^60 take the division.
template <int N>
__device__ __forceinline__ void divide_all(const double (&n)[N], double d, double (&q)[N]) {
    const unsigned h = (unsigned)__double2hiint(d);
    const int e = (int)(h >> 20 & 0x7ffu) - 1023;
    if (e <= -60 || e >= 60) {
#pragma unroll
        for (int i = 0; i < N; ++i) q[i] = n[i] / d;
        return;
    }
    const float df = __uint_as_float((h & 0x80000000u) | (unsigned)(e + 127) << 23 | (h & 0xfffffu) << 3);
    bool odd = false;  // never: 1 / df is a normal number
    const double y0 = widen_f32(__frcp_rn(df), odd);  // to 2^-22: df drops d's low bits
    double r = __fma_rn(-d, y0, 1.0);
    r = __fma_rn(r, r, r);
    const double y = __fma_rn(y0, r, y0);  // y0 (1 + r + r^2): to 2^-53
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const double t = __dmul_rn(n[i], y);
        q[i] = __fma_rn(__fma_rn(-t, d, n[i]), y, t);
    }
}

// hi + lo of a double-word sum as FP64, one FP64 operation.
__device__ __forceinline__ double widen_ff(ff x) {
    bool odd = false;
    const double h = widen_f32(x.hi, odd), l = widen_f32(x.lo, odd);
    return odd ? (double)x.hi + (double)x.lo : h + l;
}

// Sums of N = 4 or 12 values per lane over the warp.  A butterfly of every
// value is 5 N additions on every lane, and a warp's FP64 addition holds its
// scheduler's pipe for 64 clocks; here each exchange halves the values a lane
// carries instead (6 and 13 additions; the diagnostics of a 256^2 lattice,
// mostly this reduction, 19.1 -> 13.6 us).  The sum of value k is returned by
// the even lane for which warp_sum_index is k, and by its odd neighbour;
// other lanes get index N.
template <int N>
__device__ __forceinline__ int warp_sum_index(int lane) {
    if (N == 4) return lane & 18 ? N : (lane >> 3 & 1) * 2 + (lane >> 2 & 1);
    const int k = (lane >> 2 & 1) * 2 + (lane >> 1 & 1);
    return k < 3 ? (lane >> 4) * 6 + (lane >> 3 & 1) * 3 + k : N;
}
__device__ __forceinline__ double halve_sum(bool up, double lower, double upper, int o) {
    return (up ? upper : lower) + __shfl_xor_sync(0xffffffffu, up ? lower : upper, o);
}
template <int N>
__device__ __forceinline__ double warp_sum_all(const double (&v)[N], int lane) {
    static_assert(N == 4 || N == 12, "4 or 12 values");
    if constexpr (N == 12) {
        double a[6], b[3];
#pragma unroll
        for (int i = 0; i < 6; ++i) a[i] = halve_sum(lane & 16, v[i], v[6 + i], 16);
#pragma unroll
        for (int i = 0; i < 3; ++i) b[i] = halve_sum(lane & 8, a[i], a[3 + i], 8);
        const double c0 = halve_sum(lane & 4, b[0], b[2], 4), c1 = halve_sum(lane & 4, b[1], 0.0, 4);
        const double d = halve_sum(lane & 2, c0, c1, 2);
        return d + __shfl_xor_sync(0xffffffffu, d, 1);
    } else {
        const double a0 = halve_sum(lane & 8, v[0], v[2], 8), a1 = halve_sum(lane & 8, v[1], v[3], 8);
        double b = halve_sum(lane & 4, a0, a1, 4);
        b += __shfl_xor_sync(0xffffffffu, b, 16);
        b += __shfl_xor_sync(0xffffffffu, b, 2);
        return b + __shfl_xor_sync(0xffffffffu, b, 1);
    }
}

}  // namespace lbmhd

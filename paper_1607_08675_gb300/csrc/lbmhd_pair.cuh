// lbmhd_pair.cuh -- the FP32 collision with every rounding written out, of one
// node (T = float) or of two neighbouring nodes at once (T = float2) in the
// packed two-wide FP32 instructions of sm_100 and later, which take one issue
// slot for two operations.
//
// Both come from the one source below, and every FP32 step kernel calls it, so
// they give the same values whatever shape the compiler gives their code, bit
// for bit but for the sign of a zero (see mul_).  The operations are those of
// collide() (lbmhd_device.cuh) with its products fused into the sums that
// follow.  ABS: FP32 storage of the populations themselves fuses the second
// product of j_x j_y / rho - B_x B_y instead of the first; neither is the more
// accurate, and each keeps the results that its format had.  A sign moved from
// a term to a constant (n8, the outputs, -1/tau_m) changes no rounding.
#pragma once

#include <type_traits>

#include "lbmhd_device.cuh"

namespace lbmhd {

// One operation on one node (float) or on two (float2), each rounded on its own.
template <class T>
__device__ __forceinline__ T dup(float v) {
    if constexpr (std::is_same<T, float>::value) return v;
    else return make_float2(v, v);
}
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float neg_(float a) { return -a; }
__device__ __forceinline__ float abs_(float a) { return fabsf(a); }
__device__ __forceinline__ float2 add_(float2 a, float2 b) { return __fadd2_rn(a, b); }
// A product as a multiply-add of +0: ptxas fuses a packed product into a packed
// sum that follows, with their roundings written out and contraction off, but
// not a multiply-add.  A product that is -0 comes out as +0, which only a sum
// with another -0 shows: a state that holds negative zeros may come out with
// other signs of zero than from the scalar form, and with the same values.  A
// multiply-add of -0, which keeps the sign, is fused like the product (kinetic
// passes then differ in the last place).
__device__ __forceinline__ float2 mul_(float2 a, float2 b) { return __ffma2_rn(a, b, make_float2(0.0f, 0.0f)); }
__device__ __forceinline__ float2 fma_(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub_(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rc, ra, rb;\n\tmov.b64 {%0, %1}, rc;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 neg_(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ float2 abs_(float2 v) { return make_float2(fabsf(v.x), fabsf(v.y)); }
__device__ __forceinline__ float2 mul_(float k, float2 b) { return mul_(make_float2(k, k), b); }
__device__ __forceinline__ float2 fma_(float k, float2 b, float2 c) { return fma_(make_float2(k, k), b, c); }
__device__ __forceinline__ float2 rcp(float2 v) { return make_float2(rcp(v.x), rcp(v.y)); }
__device__ __forceinline__ float2 sqrt_(float2 v) { return make_float2(sqrt_(v.x), sqrt_(v.y)); }

// See collide() for the moments, rates and equilibria.
template <class T, bool SCALED, bool ABS>
__device__ __forceinline__ void collide_r(T (&d)[9], T (&g)[10], const Coll<float>& c) {
    constexpr float k1_3 = 1.0f / 3.0f, k1_6 = 1.0f / 6.0f, k5_3 = 5.0f / 3.0f;
    constexpr float k1_12 = 1.0f / 12.0f, k1_20 = 1.0f / 20.0f, k1_180 = 1.0f / 180.0f;
    const T s56 = add_(d[5], d[6]), s78 = add_(d[7], d[8]);
    const T e56 = sub_(d[5], d[6]), e13 = sub_(d[1], d[3]), e24 = sub_(d[2], d[4]);
    const T e87 = sub_(d[8], d[7]);
    const T dsum9 = add_(add_(add_(add_(d[0], d[1]), add_(d[2], d[3])),
                                   add_(add_(d[4], d[5]), add_(d[6], d[7]))), d[8]);
    const T jx = add_(add_(e13, e56), e87);
    const T jy = sub_(add_(e24, s56), s78);
    const T rho = SCALED ? fma_(c.inv_s, dsum9, dup<T>(1.0f)) : add_(dup<T>(1.0f), dsum9);
    const T irho = rcp(rho);
    const T ux = mul_(jx, irho), uy = mul_(jy, irho);
    const T bx = add_(add_(add_(g[0], g[2]), add_(g[4], g[6])), g[8]);
    const T by = add_(add_(add_(g[1], g[3]), add_(g[5], g[7])), g[9]);

    const T dsum = add_(s56, s78);
    const T m3 = sub_(e56, e87);
    const T m4 = sub_(add_(d[1], d[3]), add_(d[2], d[4]));
    const T m5 = add_(fma_(-2.0f, e13, e56), e87);
    const T m6 = sub_(fma_(-2.0f, e24, s56), s78);
    const T f0 = mul_(4.0f, d[0]);
    const T m7 = fma_(4.0f, dsum, fma_(-5.0f, add_(add_(d[1], d[2]), add_(d[3], d[4])), f0));
    const T m8 = sub_(f0, dsum);

    const T nbx = neg_(bx), njy = neg_(jy);
    T j2i = mul_(fma_(jx, jx, mul_(jy, jy)), irho);
    const T q3 = ABS ? fma_(nbx, by, mul_(mul_(jx, jy), irho)) : fma_(mul_(jx, jy), irho, mul_(nbx, by));
    const T q4 = fma_(by, by, fma_(fma_(jx, jx, mul_(njy, jy)), irho, mul_(nbx, bx)));
    T E = fma_(ux, by, mul_(uy, nbx));
    T n3, n4;
    if (SCALED) {
        j2i = mul_(c.inv_s, j2i);
        E = mul_(c.inv_s, E);
        n3 = fma_(-c.inv_s, q3, m3);
        n4 = fma_(-c.inv_s, q4, m4);
    } else {
        n3 = sub_(m3, q3);
        n4 = sub_(m4, q4);
    }
    const T n5 = add_(m5, jx), n6 = add_(m6, jy);
    const T t3 = mul_(3.0f, j2i);
    const T n7 = add_(m7, t3);
    const T n8 = add_(m8, fma_(-k5_3, dsum9, t3));

    T snu, nsm;
    if (c.les) {
        const T Q = sqrt_(fma_(4.0f, mul_(n3, n3), mul_(n4, n4)));
        const T te2 = add_(dup<T>(c.tn), sqrt_(fma_(mul_(c.k18, Q), irho, dup<T>(c.tn2))));
        snu = rcp(mul_(0.5f, te2));
        const T J = abs_(fma_(-2.0f, E, sub_(sub_(g[3], g[7]), sub_(g[4], g[8]))));
        const T tm2 = add_(dup<T>(c.te), sqrt_(fma_(c.k36, J, dup<T>(c.te2))));
        nsm = rcp(mul_(-0.5f, tm2));
    } else {
        snu = dup<T>(rcp(c.tn));
        nsm = dup<T>(rcp(-c.te));
    }
    const T s7 = c.s7 > 0.0f ? dup<T>(c.s7) : snu;
    const T s8 = c.s8 > 0.0f ? dup<T>(c.s8) : snu;

    const T a3 = mul_(0.25f, mul_(snu, n3));
    const T p4 = mul_(snu, n4), a4 = mul_(0.25f, p4), na4 = mul_(-0.25f, p4);
    const T a5 = mul_(k1_12, mul_(c.s5, n5));
    const T a6 = mul_(k1_12, mul_(c.s6, n6));
    const T a7 = mul_(k1_180, mul_(s7, n7));
    const T a8 = mul_(k1_20, mul_(s8, n8));
    const T q78 = sub_(mul_(4.0f, a7), a8);
    d[0] = fma_(-4.0f, add_(a7, a8), d[0]);
    d[1] = add_(d[1], fma_(5.0f, a7, fma_(2.0f, a5, na4)));
    d[2] = add_(d[2], fma_(5.0f, a7, fma_(2.0f, a6, a4)));
    d[3] = add_(d[3], fma_(5.0f, a7, fma_(-2.0f, a5, na4)));
    d[4] = add_(d[4], fma_(5.0f, a7, fma_(-2.0f, a6, a4)));
    const T D = sub_(a3, a5), H = sub_(a6, q78);
    d[5] = sub_(d[5], add_(add_(a3, a5), add_(a6, q78)));
    d[6] = sub_(d[6], sub_(sub_(a6, a3), sub_(a5, q78)));
    d[7] = sub_(d[7], sub_(D, H));
    d[8] = add_(d[8], add_(D, H));

    const T yp = fma_(3.0f, E, by), xm = fma_(-3.0f, E, bx);
    const T ym = fma_(-3.0f, E, by), xp = fma_(3.0f, E, bx);
    auto relax = [&](int q, float k, T v) { g[q] = fma_(nsm, fma_(-k, v, g[q]), g[q]); };
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

// A pair of nodes one after the other: for threads with more nodes, where the
// packed form's live values cost more in occupancy than its issue slots save
// (us per step, each / packed: FP32 512^2 four nodes 5.9 / 6.5, FP16 512^2 four
// nodes 4.2 / 5.0, FP16 1024^2 eight nodes 12.5 / 13.4; with two nodes packed
// wins: FP32 512^2 5.9 / 5.4, 1024^2 27.1 / 23.8, FP16 512^2 5.2 / 4.7).
template <bool SCALED, bool ABS>
__device__ __forceinline__ void collide_pair_each(float2 (&d)[9], float2 (&g)[10], const Coll<float>& c) {
    float a[9], b[10];
#pragma unroll
    for (int i = 0; i < 9; ++i) a[i] = d[i].x;
#pragma unroll
    for (int q = 0; q < 10; ++q) b[q] = g[q].x;
    collide_r<float, SCALED, ABS>(a, b, c);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        d[i].x = a[i];
        a[i] = d[i].y;
    }
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        g[q].x = b[q];
        b[q] = g[q].y;
    }
    collide_r<float, SCALED, ABS>(a, b, c);
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i].y = a[i];
#pragma unroll
    for (int q = 0; q < 10; ++q) g[q].y = b[q];
}

// ---- the kinetic closures --------------------------------------------------
// collide_xf, filtered_shift, carati_taus and the moment sums of
// lbmhd_kinetic.cu (a file compiled without contraction) with every rounding
// written out: the same operations in the same order, so the same values.
__device__ __forceinline__ float recip_(float v) { return __frcp_rn(v); }
__device__ __forceinline__ float2 recip_(float2 v) { return make_float2(__frcp_rn(v.x), __frcp_rn(v.y)); }
__device__ __forceinline__ float root_(float v) { return __fsqrt_rn(v); }
__device__ __forceinline__ float2 root_(float2 v) { return make_float2(__fsqrt_rn(v.x), __fsqrt_rn(v.y)); }
__device__ __forceinline__ float sign_(float v) { return v > 0.0f ? 1.0f : (v < 0.0f ? -1.0f : 0.0f); }
__device__ __forceinline__ float2 sign_(float2 v) { return make_float2(sign_(v.x), sign_(v.y)); }
__device__ __forceinline__ float least_half_(float v) { return v < 0.5f ? 0.5f : v; }
__device__ __forceinline__ float2 least_half_(float2 v) { return make_float2(least_half_(v.x), least_half_(v.y)); }

// rho, jx, jy, Bx, By of decoded streamed populations.
template <class T, bool SCALED>
__device__ __forceinline__ void moments_r(const T (&d)[9], const T (&g)[10], float inv_s, T (&m)[5]) {
    T drho = add_(add_(add_(add_(d[0], d[1]), add_(d[2], d[3])),
                       add_(add_(d[4], d[5]), add_(d[6], d[7]))), d[8]);
    m[1] = add_(add_(sub_(d[1], d[3]), sub_(d[5], d[6])), sub_(d[8], d[7]));
    m[2] = sub_(add_(sub_(d[2], d[4]), add_(d[5], d[6])), add_(d[7], d[8]));
    m[3] = add_(add_(add_(g[0], g[2]), add_(g[4], g[6])), g[8]);
    m[4] = add_(add_(add_(g[1], g[3]), add_(g[5], g[7])), g[9]);
    if (SCALED) {
        drho = mul_(inv_s, drho);
#pragma unroll
        for (int q = 1; q < 5; ++q) m[q] = mul_(inv_s, m[q]);
    }
    m[0] = add_(dup<T>(1.0f), drho);
}

template <class T>
__device__ __forceinline__ void filtered_shift_r(const T (&f)[5], const T (&gx)[5], const T (&gy)[5],
                                                 float d2, T (&sh)[4]) {
    const T ir = recip_(f[0]);
    constexpr float twelfth = 1.0f / 12.0f;
    const T scale = mul_(ir, dup<T>(twelfth));
    auto dot = [&](int a, int b) { return add_(mul_(gx[a], gx[b]), mul_(gy[a], gy[b])); };
    T d0[5];
#pragma unroll
    for (int a = 0; a < 5; ++a) d0[a] = dot(0, a);
    auto ratio = [&](int a, int b) {
        const T in = sub_(add_(mul_(f[a], d0[b]), mul_(f[b], d0[a])), mul_(mul_(mul_(f[a], f[b]), d0[0]), ir));
        return mul_(sub_(dot(a, b), mul_(in, ir)), scale);
    };
    const T rxx = ratio(1, 1), ryy = ratio(2, 2), rxy = ratio(1, 2);
    sh[0] = mul_(d2, sub_(rxy, mul_(twelfth, dot(3, 4))));
    sh[1] = mul_(d2, sub_(sub_(rxx, ryy), mul_(twelfth, sub_(dot(3, 3), dot(4, 4)))));
    sh[2] = mul_(d2, mul_(-3.0f, add_(rxx, ryy)));
    sh[3] = mul_(d2, sub_(ratio(1, 4), ratio(2, 3)));
}

// gu, gb: d/dx, d/dy of (u_x, u_y) and (B_x, B_y).
template <class T>
__device__ __forceinline__ void carati_taus_r(const T (&gu)[2][2], const T (&gb)[2][2],
                                              const Coll<float>& c, T (&taus)[2]) {
    const T svxy = mul_(0.5f, add_(gu[0][1], gu[1][0])), sbxy = mul_(0.5f, add_(gb[0][1], gb[1][0]));
    const T ss = add_(add_(mul_(gu[0][0], gb[0][0]), mul_(gu[1][1], gb[1][1])), mul_(mul_(2.0f, svxy), sbxy));
    const T nu_t = mul_(c.cd2, root_(abs_(ss)));
    const T jw = mul_(sub_(gb[1][0], gb[0][1]), sub_(gu[1][0], gu[0][1]));
    const T eta_t = mul_(mul_(c.cd2, sign_(jw)), root_(abs_(jw)));
    taus[0] = add_(dup<T>(c.tn), mul_(3.0f, nu_t));
    taus[1] = least_half_(add_(dup<T>(c.te), mul_(3.0f, eta_t)));
}

// KIN: sh = corrections of M_3, M_4, M_7 = M_8, N_y1 (les 2); else sh[0], sh[1]
// are the relaxation times (les 3).
template <class T, bool SCALED, bool KIN>
__device__ __forceinline__ void collide_kin_r(T (&d)[9], T (&g)[10], const Coll<float>& c, const T* sh) {
    constexpr float k1_3 = 1.0f / 3.0f, k1_6 = 1.0f / 6.0f, k5_3 = 5.0f / 3.0f;
    constexpr float k1_12 = 1.0f / 12.0f, k1_20 = 1.0f / 20.0f, k1_180 = 1.0f / 180.0f;
    const T s56 = add_(d[5], d[6]), s78 = add_(d[7], d[8]);
    const T e56 = sub_(d[5], d[6]), e87 = sub_(d[8], d[7]), e13 = sub_(d[1], d[3]), e24 = sub_(d[2], d[4]);
    const T dsum9 = add_(add_(add_(add_(d[0], d[1]), add_(d[2], d[3])),
                              add_(add_(d[4], d[5]), add_(d[6], d[7]))), d[8]);
    const T jx = add_(add_(e13, e56), e87), jy = sub_(add_(e24, s56), s78);
    const T rho = SCALED ? fma_(c.inv_s, dsum9, dup<T>(1.0f)) : add_(dup<T>(1.0f), dsum9);
    const T irho = rcp(rho);
    const T ux = mul_(jx, irho), uy = mul_(jy, irho);
    const T bx = add_(add_(add_(g[0], g[2]), add_(g[4], g[6])), g[8]);
    const T by = add_(add_(add_(g[1], g[3]), add_(g[5], g[7])), g[9]);
    const T dsum = add_(s56, s78);
    const T m3 = sub_(e56, e87), m4 = sub_(add_(d[1], d[3]), add_(d[2], d[4]));
    const T m5 = fma_(-2.0f, e13, add_(e56, e87)), m6 = fma_(-2.0f, e24, sub_(s56, s78));
    const T m7 = fma_(-5.0f, add_(add_(d[1], d[2]), add_(d[3], d[4])), mul_(4.0f, add_(d[0], dsum)));
    const T m8 = sub_(mul_(4.0f, d[0]), dsum);
    const T nbx = neg_(bx), njy = neg_(jy);
    T j2i = mul_(fma_(jx, jx, mul_(jy, jy)), irho);
    T q3 = fma_(mul_(jx, jy), irho, mul_(nbx, by));
    T q4 = fma_(fma_(jx, jx, mul_(njy, jy)), irho, fma_(by, by, mul_(nbx, bx)));
    T E = fma_(ux, by, mul_(uy, nbx));
    if (SCALED) {
        j2i = mul_(c.inv_s, j2i);
        q3 = mul_(c.inv_s, q3);
        q4 = mul_(c.inv_s, q4);
        E = mul_(c.inv_s, E);
    }
    if (KIN) {
        q3 = add_(q3, sh[0]);
        q4 = add_(q4, sh[1]);
        E = add_(E, sh[3]);
    }
    const T n3 = sub_(m3, q3), n4 = sub_(m4, q4), n5 = add_(m5, jx), n6 = add_(m6, jy);
    T n7 = fma_(3.0f, j2i, m7), x8 = fma_(k5_3, dsum9, mul_(-3.0f, j2i));
    if (KIN) {
        n7 = sub_(n7, sh[2]);
        x8 = add_(x8, sh[2]);
    }
    const T n8 = sub_(m8, x8);
    const T snu = KIN ? dup<T>(rcp(c.tn)) : rcp(sh[0]);
    const T nsm = KIN ? dup<T>(-rcp(c.te)) : neg_(rcp(sh[1]));
    const T s7 = c.s7 > 0.0f ? dup<T>(c.s7) : snu, s8 = c.s8 > 0.0f ? dup<T>(c.s8) : snu;
    const T a3 = mul_(0.25f, mul_(snu, n3));
    const T p4 = mul_(snu, n4), a4 = mul_(0.25f, p4), na4 = mul_(-0.25f, p4);
    const T a5 = mul_(k1_12, mul_(c.s5, n5)), a6 = mul_(k1_12, mul_(c.s6, n6));
    const T a7 = mul_(k1_180, mul_(s7, n7)), a8 = mul_(k1_20, mul_(s8, n8));
    const T q78 = sub_(mul_(4.0f, a7), a8);
    d[0] = fma_(-4.0f, add_(a7, a8), d[0]);
    d[1] = add_(d[1], fma_(5.0f, a7, fma_(2.0f, a5, na4)));
    d[2] = add_(d[2], fma_(5.0f, a7, fma_(2.0f, a6, a4)));
    d[3] = add_(d[3], fma_(5.0f, a7, fma_(-2.0f, a5, na4)));
    d[4] = add_(d[4], fma_(5.0f, a7, fma_(-2.0f, a6, a4)));
    const T D = sub_(a3, a5), H = sub_(a6, q78);
    d[5] = sub_(d[5], add_(add_(a3, a5), add_(a6, q78)));
    d[6] = sub_(d[6], sub_(sub_(a6, a3), sub_(a5, q78)));
    d[7] = sub_(d[7], sub_(D, H));
    d[8] = add_(d[8], add_(D, H));
    const T e3 = mul_(3.0f, E), bx6 = mul_(k1_6, bx), by6 = mul_(k1_6, by);
    auto relax = [&](int q, T eq) { g[q] = fma_(nsm, sub_(g[q], eq), g[q]); };
    relax(0, mul_(k1_3, bx));
    relax(1, mul_(k1_3, by));
    relax(2, bx6);
    relax(3, mul_(k1_6, add_(by, e3)));
    relax(4, mul_(k1_6, sub_(bx, e3)));
    relax(5, by6);
    relax(6, bx6);
    relax(7, mul_(k1_6, sub_(by, e3)));
    relax(8, mul_(k1_6, add_(bx, e3)));
    relax(9, by6);
}

}  // namespace lbmhd

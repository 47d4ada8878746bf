// pond_vec.cuh -- the arithmetic of the lane kernels, written once for FP64 and for packed
// FP32.
//
// FP32 kernels carry two faces per thread, one in each lane of the FP32x2 instructions of
// sm_100 and later (Lane2): both faces run the same operations on their own data, so every
// multiply-add serves two and no operand has to be broadcast or paired up.  FP64 kernels
// carry one face per thread (double).  The code between the two is the same template.  Lane2 operations
// round where they say (each is one instruction); in scalar code of the same templates, in FP64 and in the FP32
// tails, the compiler may contract a product that is not written as vfma into a sum.
#pragma once

#include "pond_core.cuh"

namespace pond {

struct Lane2 {
    float2 v;
};

template <typename R> struct VecOf;
template <> struct VecOf<float> { using type = Lane2; static constexpr int lanes = 2; };
template <> struct VecOf<double> { using type = double; static constexpr int lanes = 1; };

template <typename V> __device__ __forceinline__ V vset(double c);   // a constant in every lane
template <> __device__ __forceinline__ Lane2 vset<Lane2>(double c) { return Lane2{make_float2(float(c), float(c))}; }
template <> __device__ __forceinline__ double vset<double>(double c) { return c; }
template <> __device__ __forceinline__ float vset<float>(double c) { return float(c); }
__device__ __forceinline__ Lane2 vbc(float c) { return Lane2{make_float2(c, c)}; }
__device__ __forceinline__ double vbc(double c) { return c; }

__device__ __forceinline__ Lane2 operator+(Lane2 a, Lane2 b) { return Lane2{__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ Lane2 operator*(Lane2 a, Lane2 b) { return Lane2{__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ Lane2 operator-(Lane2 a, Lane2 b)
{
    return Lane2{__fadd2_rn(a.v, make_float2(-b.v.x, -b.v.y))};
}
__device__ __forceinline__ Lane2 vfma(Lane2 a, Lane2 b, Lane2 c) { return Lane2{__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }

// a product that no sum may absorb
__device__ __forceinline__ double vmul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float vmul_rn(float a, float b) { return __fmul_rn(a, b); }

// the lane l (0 or 1) of a value
__device__ __forceinline__ float vget(const Lane2 &a, int l) { return l ? a.v.y : a.v.x; }
__device__ __forceinline__ double vget(const double &a, int) { return a; }
__device__ __forceinline__ void vput(Lane2 &a, int l, float x)
{
    if (l) a.v.y = x;
    else a.v.x = x;
}
__device__ __forceinline__ void vput(double &a, int, double x) { a = x; }
__device__ __forceinline__ void vput(float &a, int, float x) { a = x; }

__device__ __forceinline__ Lane2 vsqrt(Lane2 a) { return Lane2{make_float2(w_sqrt<float>(a.v.x), w_sqrt<float>(a.v.y))}; }
__device__ __forceinline__ double vsqrt(double a) { return sqrt(a); }
__device__ __forceinline__ float vsqrt(float a) { return w_sqrt<float>(a); }
__device__ __forceinline__ Lane2 vrcp(Lane2 a) { return Lane2{make_float2(w_rcp<float>(a.v.x), w_rcp<float>(a.v.y))}; }
__device__ __forceinline__ double vrcp(double a) { return 1.0 / a; }
__device__ __forceinline__ float vrcp(float a) { return w_rcp<float>(a); }

// ---- limited slopes, divided by 2 for van Leer (ab/(a+b) where ab > 0, else 0; the factor is
// exact and goes into the departure offsets) and as they are for minmod
__device__ __forceinline__ float rcp_ftz(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// Where ab > 0 in FP32, |a + b| is at least 2^-75: a normal number, for which the flush-to-zero
// reciprocal is the plain one without its range test.
__device__ __forceinline__ Lane2 vanleer_half(Lane2 a, Lane2 b)
{
    const Lane2 ab = a * b, s = a + b;
    const Lane2 q = ab * Lane2{make_float2(rcp_ftz(s.v.x), rcp_ftz(s.v.y))};
    return Lane2{make_float2(ab.v.x > 0.f ? q.v.x : 0.f, ab.v.y > 0.f ? q.v.y : 0.f)};
}
__device__ __forceinline__ float vanleer_half(float a, float b)
{
    const float ab = a * b;
    return ab > 0.f ? ab * rcp_ftz(a + b) : 0.f;
}
// FP64: the quotient from the hardware's 20-bit reciprocal of a + b, one Newton step on it and one on the quotient
// (q = q0 + r1 (ab - s q0), q0 = ab r0, r1 = r0 (2 - s r0)): the residual is exact to 2^-73 of ab and r1 to
// 2^-38, so q is within 2^-57 of ab / s before its one rounding, as good as the division.  The test ab > 0 is
// on the sign and exponent bits.  GB300 runs FP64 at 1/64 of the FP32 rate, and the
// corrector evaluates this 64 times a pass in 2D and 384 times in 3D.  Where ab > 0, |a + b| is
// above 2^-522, so the seed's flush of subnormals does not matter.
__device__ __forceinline__ double vanleer_half(double a, double b)
{
    const double ab = a * b, s = a + b;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s));
    const double q0 = __dmul_rn(ab, r), r1 = fma(r, fma(-s, r, 1.0), r);
    const double q = fma(fma(-s, q0, ab), r1, q0);
    // 0 < high word <= that of infinity: positive, not NaN
    return unsigned(__double2hiint(ab) - 1) < 0x7ff00000u ? q : 0.0;
}
__device__ __forceinline__ Lane2 vminmod(Lane2 a, Lane2 b)
{
    return Lane2{make_float2(minmod<float>(a.v.x, b.v.x), minmod<float>(a.v.y, b.v.y))};
}
__device__ __forceinline__ double vminmod(double a, double b) { return minmod<double>(a, b); }
__device__ __forceinline__ float vminmod(float a, float b) { return minmod<float>(a, b); }

// ---- (f, g) pairs: f in lane x and g in lane y of packed FP32x2 instructions in FP32 (worth it where
// the multiplier is a node constant), two words in FP64
template <typename R> struct FG;
template <> struct FG<float> { float2 v; };
template <> struct FG<double> { double f, g; };
__device__ __forceinline__ FG<float> fg(float f, float g) { return {make_float2(f, g)}; }
__device__ __forceinline__ FG<double> fg(double f, double g) { return {f, g}; }
__device__ __forceinline__ FG<float> operator+(FG<float> a, FG<float> b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ FG<double> operator+(FG<double> a, FG<double> b) { return {a.f + b.f, a.g + b.g}; }
__device__ __forceinline__ FG<float> operator-(FG<float> a, FG<float> b) { return {__fadd2_rn(a.v, make_float2(-b.v.x, -b.v.y))}; }
__device__ __forceinline__ FG<double> operator-(FG<double> a, FG<double> b) { return {a.f - b.f, a.g - b.g}; }
__device__ __forceinline__ FG<float> operator*(FG<float> a, float c) { return {__fmul2_rn(a.v, make_float2(c, c))}; }
__device__ __forceinline__ FG<double> operator*(FG<double> a, double c) { return {a.f * c, a.g * c}; }
__device__ __forceinline__ FG<float> fgfma(FG<float> a, float c, FG<float> b) { return {__ffma2_rn(a.v, make_float2(c, c), b.v)}; }
__device__ __forceinline__ FG<double> fgfma(FG<double> a, double c, FG<double> b) { return {fma(a.f, c, b.f), fma(a.g, c, b.g)}; }
__device__ __forceinline__ float fpart(const FG<float> &a) { return a.v.x; }
__device__ __forceinline__ float gpart(const FG<float> &a) { return a.v.y; }
__device__ __forceinline__ double fpart(const FG<double> &a) { return a.f; }
__device__ __forceinline__ double gpart(const FG<double> &a) { return a.g; }
// the f part increased by x c
__device__ __forceinline__ void add_f(FG<float> &a, float x, float c) { a.v.x = fmaf(x, c, a.v.x); }
__device__ __forceinline__ void add_f(FG<double> &a, double x, double c) { a.f = fma(x, c, a.f); }
__device__ __forceinline__ FG<float> vanleer_half(FG<float> a, FG<float> b) { return {vanleer_half(Lane2{a.v}, Lane2{b.v}).v}; }
__device__ __forceinline__ FG<double> vanleer_half(FG<double> a, FG<double> b)
{
    return {vanleer_half(a.f, b.f), vanleer_half(a.g, b.g)};
}
__device__ __forceinline__ FG<float> vminmod(FG<float> a, FG<float> b) { return {vminmod(Lane2{a.v}, Lane2{b.v}).v}; }
__device__ __forceinline__ FG<double> vminmod(FG<double> a, FG<double> b) { return {vminmod(a.f, b.f), vminmod(a.g, b.g)}; }
__device__ __forceinline__ FG<double> fgsel(bool c, FG<double> a, FG<double> b) { return {c ? a.f : b.f, c ? a.g : b.g}; }

// ---- the regularized change of frame (Sec. II.C) in shift form
//
// With s = sqrt(T/T'), e = s^2 - 1 and d = (u - u')/sqrt(T') per axis, the products of the
// one-dimensional maps (pond_core.cuh) collapse to recurrences in the new coefficients: an
// order follows from the one below by a multiplication with d, and no map entry is formed.
// For coefficients in the frame of their own first moment (f, first order zero):
//     F_10 = dx A,           q_x = e A + s^2 A_20,  F_20 = dx F_10 + q_x,
//     F_11 = dx F_01 + a11,  F_30 = dx (F_20 + 2 q_x) + s^3 A_30,
//     F_21 = dy F_20 + 2 dx a11 + s^3 A_21          (a11 = s^2 A_11)
// and the same with the axes exchanged: 25 operations in 2D, against 45 for the maps and
// their products.  The identity (d = e = 0) stays exact.
template <typename R>
struct Move1 {
    R s, e, d, s2, s3;
    __device__ __forceinline__ Move1(R s_, R e_, R d_) : s(s_), e(e_), d(d_), s2(e_ + R(1)), s3(s2 * s_) {}
    // orders 0..3 and 0..2, with a first order
    __device__ __forceinline__ void f(const R *A, R *F) const
    {
        const R a1 = s * A[1], q = vfma(s2, A[2], e * A[0]);
        F[0] = A[0];
        F[1] = vfma(d, A[0], a1);
        F[2] = vfma(d, F[1] + a1, q);
        F[3] = vfma(s3, A[3], vfma(R(3) * e, a1, d * vfma(d, a1, vfma(R(2), q, F[2]))));
    }
    __device__ __forceinline__ void g(const R *B, R *G) const
    {
        const R b1 = s * B[1];
        G[0] = B[0];
        G[1] = vfma(d, B[0], b1);
        G[2] = vfma(d, G[1] + b1, vfma(s2, B[2], e * B[0]));
    }
};

template <typename V>
struct Move2 {
    V s, e, dx, dy, s2, s3;
    // Tc, cx, cy: the cell's frame; Tl, (lx, ly): the target frame, velocities on one reference
    __device__ __forceinline__ Move2(V Tc, V cx, V cy, V Tl, V invTl, V rsqTl, V lx, V ly)
    {
        s = vsqrt(Tc * invTl);
        e = (Tc - Tl) * invTl;
        dx = (cx - lx) * rsqTl;
        dy = (cy - ly) * rsqTl;
        s2 = e + vset<V>(1.0);
        s3 = s2 * s;
    }
    // first order zero -> F[10] in hidx order
    __device__ __forceinline__ void f(V A00, V A20, V A11, V A02, V A30, V A21, V A12, V A03, V *F) const
    {
        const V e0 = e * A00, dx2 = dx + dx, dy2 = dy + dy, two = vset<V>(2.0);
        F[0] = A00;
        F[hidx(1, 0)] = dx * A00;
        F[hidx(0, 1)] = dy * A00;
        const V qx = vfma(s2, A20, e0), qy = vfma(s2, A02, e0), a11 = s2 * A11;
        F[hidx(2, 0)] = vfma(dx, F[hidx(1, 0)], qx);
        F[hidx(0, 2)] = vfma(dy, F[hidx(0, 1)], qy);
        F[hidx(1, 1)] = vfma(dx, F[hidx(0, 1)], a11);
        F[hidx(2, 1)] = vfma(s3, A21, vfma(dx2, a11, dy * F[hidx(2, 0)]));
        F[hidx(1, 2)] = vfma(s3, A12, vfma(dy2, a11, dx * F[hidx(0, 2)]));
        F[hidx(3, 0)] = vfma(s3, A30, dx * vfma(two, qx, F[hidx(2, 0)]));
        F[hidx(0, 3)] = vfma(s3, A03, dy * vfma(two, qy, F[hidx(0, 2)]));
    }
    // the same for coefficients with a first order (hidx order)
    __device__ __forceinline__ void f_full(const V *A, V *F) const
    {
        const V a10 = s * A[1], a01 = s * A[2], e0 = e * A[0], two = vset<V>(2.0), three = vset<V>(3.0);
        const V ex = vfma(dx, dx, e), ey = vfma(dy, dy, e);
        F[0] = A[0];
        F[1] = vfma(dx, A[0], a10);
        F[2] = vfma(dy, A[0], a01);
        const V qx = vfma(s2, A[3], e0), qy = vfma(s2, A[5], e0), a11 = s2 * A[4];
        F[3] = vfma(dx, F[1] + a10, qx);
        F[5] = vfma(dy, F[2] + a01, qy);
        F[4] = vfma(dx, F[2], vfma(dy, a10, a11));
        F[hidx(2, 1)] = vfma(s3, A[7], vfma(dx + dx, a11, vfma(ex, a01, dy * F[3])));
        F[hidx(1, 2)] = vfma(s3, A[8], vfma(dy + dy, a11, vfma(ey, a10, dx * F[5])));
        F[hidx(3, 0)] = vfma(s3, A[6], vfma(three * e, a10, dx * vfma(dx, a10, vfma(two, qx, F[3]))));
        F[hidx(0, 3)] = vfma(s3, A[9], vfma(three * e, a01, dy * vfma(dy, a01, vfma(two, qy, F[5]))));
    }
    // the six coefficients of order <= 2 -> G in hidx order
    __device__ __forceinline__ void g(V B00, V B10, V B01, V B20, V B11, V B02, V *G) const
    {
        const V b10 = s * B10, b01 = s * B01, e0 = e * B00;
        G[0] = B00;
        G[1] = vfma(dx, B00, b10);
        G[2] = vfma(dy, B00, b01);
        G[3] = vfma(dx, G[1] + b10, vfma(s2, B20, e0));
        G[5] = vfma(dy, G[2] + b01, vfma(s2, B02, e0));
        G[4] = vfma(s2, B11, vfma(dy, b10, dx * G[2]));
    }
};

}  // namespace pond

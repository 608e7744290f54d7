// Round-robin schedule and plane rotations, shared by the two-sided eigensolver
// (jacobi.cu) and the one-sided SVT solver (osj.cu).
#pragma once
#include "common.cuh"

namespace lrr {

// item at position `pos` of round `r` in the circle-method schedule of N items:
// every round pairs position k with N-1-k, and N-1 rounds pair every two items once
__device__ __forceinline__ int circle_item(int pos, int r, int N) {
    return pos == 0 ? 0 : 1 + ((pos - 1 + r) % (N - 1));
}

// Rotation (c, s) that annihilates s_pq: tan(2 theta) = 2 s_pq / (s_qq - s_pp),
// the tangent's root of smaller magnitude.
template <typename T>
__device__ __forceinline__ void jacobi_rotation(T app, T aqq, T apq, T& cc, T& ss);

// float64 quotients, reciprocals and square roots of the rotation, rounded as
// IEEE division and square root round them.  Three divisions and two square
// roots in a chain were 60 % of the float64 pivots; here each starts from the
// float32 unit's approximation, takes one Newton step in float64 and ends with
// the remainder correction of P. Markstein ("IA-64 and Elementary Functions",
// 2000, ch. 8 and 9).  The result before its last rounding is good to 2^-88 or
// better, so it differs from the IEEE one with probability below 2^-34.
// (Equal in 4e9 random cases each, tested against / and sqrt.)

// 1 / b (1 + O(2^-45)) for b whose float32 reciprocal is normal
__device__ __forceinline__ double rcp_newton(double b) {
    float f;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((float)b));
    const double y = (double)f;
    return fma(y, fma(-b, y, 1.0), y);
}
// 1 / b
__device__ __forceinline__ double rcp_rn(double b, double y) { return fma(y, fma(-b, y, 1.0), y); }
// a / b over the whole range: mantissas in [1, 2) and the exponents apart; near
// the ends of the range the division itself
__device__ __forceinline__ double div_rn(double a, double b) {
    const int ha = __double2hiint(a), hb = __double2hiint(b);
    const int ea = (ha >> 20) & 0x7FF, eb = (hb >> 20) & 0x7FF;
    const int n = ea - eb;
    if (ea < 64 || ea > 1982 || eb < 64 || eb > 1982 || n > 900 || n < -900) return a / b;
    const double am = __hiloint2double((ha & 0x000FFFFF) | 0x3FF00000, __double2loint(a));
    const double bm = __hiloint2double((hb & 0x000FFFFF) | 0x3FF00000, __double2loint(b));
    const double y = rcp_newton(bm);
    const double q = am * y;
    const double r = fma(fma(-bm, q, am), y, q);
    return r * __hiloint2double(((ha ^ hb) & 0x80000000) | ((n + 1023) << 20), 0);
}
// s = sqrt(x) and y = 1 / s (1 + O(2^-43)), x in [1, 1e32]
__device__ __forceinline__ double sqrt_rn(double x, double& y) {
    float f;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((float)x));
    const double y0 = (double)f, g = x * y0, h = 0.5 * y0;
    const double r = fma(-h, g, 0.5);
    const double g1 = fma(g, r, g), h1 = fma(h, r, h);
    y = 2.0 * h1;
    return fma(fma(-g1, g1, x), h1, g1);
}
template <>
__device__ __forceinline__ void jacobi_rotation<double>(double app, double aqq, double apq, double& cc, double& ss) {
    const double theta = div_rn(aqq - app, 2.0 * apq);
    double tt, y;
    if (fabs(theta) > 1.0 / DBL_EPSILON) {
        tt = div_rn(0.5, theta);
    } else {
        const double b = fabs(theta) + sqrt_rn(fma(theta, theta, 1.0), y);
        const double t = rcp_rn(b, rcp_newton(b));
        tt = theta >= 0.0 ? t : -t;
    }
    const double h = sqrt_rn(fma(tt, tt, 1.0), y);
    cc = rcp_rn(h, y);
    ss = tt * cc;
}
// float: the hardware reciprocal and reciprocal square root.  The rotations
// only steer the pivot towards diagonal form: the accumulated rotation is
// re-orthonormalised before it touches the columns, and the next sweep forms
// its Grams afresh, so a few ulps in c and s cost no accuracy, while the
// shorter dependent chain shortens every step of the inner sweep.
template <>
__device__ __forceinline__ void jacobi_rotation<float>(float app, float aqq, float apq, float& cc, float& ss) {
    const float theta = __fdividef(aqq - app, 2.f * apq);
    float tt;
    if (fabsf(theta) > 1.f / FLT_EPSILON) {
        tt = __fdividef(0.5f, theta);
    } else {
        const float h = fmaf(theta, theta, 1.f);
        tt = copysignf(__fdividef(1.f, fabsf(theta) + h * rsqrtf(h)), theta);
    }
    cc = rsqrtf(fmaf(tt, tt, 1.f));
    ss = tt * cc;
}

}  // namespace lrr

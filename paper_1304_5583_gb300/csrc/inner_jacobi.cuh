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

// off > eps sqrt(g) exactly (g >= 0): the rounded root, some 40 dependent cycles and
// a branch of its own, only where the hardware's approximation does not decide
__device__ __forceinline__ bool above_eps_root(float off, float g) {
    const bool low = g < 1e-30f;             // (subnormal products are common: scaled, exactly)
    float q;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(low ? g * 0x1p100f : g));
    const float bound = (low ? 0x1p-50f * FLT_EPSILON : FLT_EPSILON) * q;
    if (off > 1.0001f * bound || off < 0.9999f * bound) return off > bound;
    return off > FLT_EPSILON * sqrtf(g);
}

// Rotation (c, s) that annihilates s_pq: tan(2 theta) = 2 s_pq / (s_qq - s_pp),
// the tangent's root of smaller magnitude.
template <typename T>
__device__ __forceinline__ void jacobi_rotation(T app, T aqq, T apq, T& cc, T& ss);

// float64 quotients, reciprocals and square roots of the rotation, rounded as
// IEEE division and square root round them but for one in 2^30.  A dependent float64 operation takes
// 65 cycles here (a float32 one 4), conversions and compares included, so the
// seeds are taken to 2^-43 in pairs of float32 (one Newton step on the hardware
// approximation, the argument's low bits as a second float32), exponents and
// conversions are handled as integers, and float64 is left with the product and
// the remainder correction of P. Markstein ("IA-64 and Elementary Functions",
// 2000, ch. 8 and 9): 3 operations for a quotient or a root, 2 for a
// reciprocal.  The result before its last rounding is good to 2^-84 (1.5 e^2 for
// a root, e^2 otherwise, with seeds good to e = 2^-42.7), so it may differ from
// the IEEE one, in the last bit, only where the exact value lies that close to
// the middle between two float64 values.
// (4e9 random cases each against / and sqrt: one reciprocal differed.)

// y0 + y1 as a double, for y0 in [0.5, 1], |y1| < 2^-21, to 2^-44: y1 is added
// to the bit pattern in units of 2^-43 (2^10 units in the last place)
__device__ __forceinline__ double join(float y0, float y1) {
    const int k = __float_as_int(fmaf(y1, 8796093022208.f, 12582912.f)) - 0x4B400000;
    const int f = __float_as_int(y0);
    const long long bits = (long long)(((unsigned long long)(unsigned)((f >> 3) + 0x38000000) << 32) | ((unsigned)f << 29));
    return __longlong_as_double(bits + ((long long)k << 10));
}
// mantissa of b (high word hb, low word lb) as high + low 2^-23, high in [1, 2)
__device__ __forceinline__ void split_mantissa(int hb, int lb, float& high, float& low) {
    high = __int_as_float(0x3F800000 | ((hb & 0x000FFFFF) << 3) | (int)((unsigned)lb >> 29));
    low = __int_as_float(0x3F800000 | (int)(((unsigned)lb << 3) >> 9)) - 1.f;
}
// 2^n b for a result in the normal range
__device__ __forceinline__ double scale2(double b, int n) {
    return __hiloint2double(__double2hiint(b) + (n << 20), __double2loint(b));
}
// 1 / m (1 + O(2^-43)), m in [1, 2) the mantissa of (hb, lb)
__device__ __forceinline__ double rcp_seed(int hb, int lb) {
    float bh, bl, y;
    split_mantissa(hb, lb, bh, bl);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(bh));
    y = fmaxf(y, 0.5f);
    const float e = fmaf(bl, y * -0x1p-23f, fmaf(-bh, y, 1.f));
    return join(y, y * fmaf(e, e, e));
}
// 1 / s from y = (1 / s)(1 + O(2^-43))
__device__ __forceinline__ double rcp_rn(double s, double y) { return fma(y, fma(-s, y, 1.0), y); }
// 1 / b, b in [1, 2^900].  A mantissa of ones, which sums at 2^53 have, is the one
// whose reciprocal 2^k (1 + 2^-53 + 2^-106) lies nearest to a middle: its last
// bit is set.  (A cosine's root, below 1.5, has no such mantissa.)
__device__ __forceinline__ double rcp_rn(double b) {
    const int hb = __double2hiint(b), lb = __double2loint(b);
    const double r = rcp_rn(b, scale2(rcp_seed(hb, lb), 1023 - (hb >> 20)));
    return __hiloint2double(__double2hiint(r), __double2loint(r) | (((hb | 0xFFF00000) & lb) == -1));
}
// a / b over the whole range: mantissas in [1, 2) and the exponents apart; near
// the ends of the range the division itself
__device__ __forceinline__ double div_rn(double a, double b) {
    const int ha = __double2hiint(a), hb = __double2hiint(b), lb = __double2loint(b);
    const int ea = (ha >> 20) & 0x7FF, eb = (hb >> 20) & 0x7FF;
    const int n = ea - eb;
    if (ea < 64 || ea > 1982 || eb < 64 || eb > 1982 || n > 900 || n < -900) return a / b;
    const double am = __hiloint2double((ha & 0x000FFFFF) | 0x3FF00000, __double2loint(a));
    const double bm = __hiloint2double((hb & 0x000FFFFF) | 0x3FF00000, lb);
    const double y = rcp_seed(hb, lb);
    const double q = am * y;
    const double r = fma(fma(-bm, q, am), y, q);
    return __hiloint2double((__double2hiint(r) + (n << 20)) | ((ha ^ hb) & 0x80000000), __double2loint(r));
}
// s = sqrt(x) and y = 1 / s (1 + O(2^-43)), x in [1, 1e32]
__device__ __forceinline__ double sqrt_rn(double x, double& y) {
    const int hx = __double2hiint(x), lx = __double2loint(x), ex = (hx >> 20) - 1023;
    float mh, ml, r;
    split_mantissa(hx, lx, mh, ml);                 // x = (mh + 2^-23 ml) 2^ex
    if (ex & 1) { mh += mh; ml += ml; }             // now in [1, 4), and an even power
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(mh));
    r = fmaxf(r, 0.5f);
    const float p = r * r, pl = fmaf(r, r, -p);     // r^2 = p + pl
    const float e = fmaf(ml, p * -0x1p-23f, fmaf(-mh, pl, fmaf(-mh, p, 1.f)));
    y = scale2(join(r, r * e * fmaf(0.375f, e, 0.5f)), -(ex >> 1));
    const double g = x * y;
    return fma(fma(-g, g, x), scale2(y, -1), g);
}
template <>
__device__ __forceinline__ void jacobi_rotation<double>(double app, double aqq, double apq, double& cc, double& ss) {
    // tan = 1 / (|theta| + sqrt(theta^2 + 1)), beyond 1 / eps 1 / (2 |theta|): one
    // reciprocal either way, so that lanes of both kinds share it
    const double theta = div_rn(aqq - app, 2.0 * apq);
    const int ht = __double2hiint(theta) & 0x7FFFFFFF, lt = __double2loint(theta);
    const int sign = __double2hiint(theta) < 0 && (ht | lt) != 0 ? (int)0x80000000 : 0;
    const bool large = ht > 0x43300000 || (ht == 0x43300000 && lt != 0);        // |theta| > 2^52
    const double at = __hiloint2double(ht, lt);
    double tt, y;
    if (ht < (1023 + 900) << 20) {
        const double sum = at + sqrt_rn(fma(theta, theta, 1.0), y);
        const double t = rcp_rn(large ? at : sum);
        tt = __hiloint2double((__double2hiint(t) - (large ? 1 << 20 : 0)) | sign, __double2loint(t));
    } else {
        tt = 0.5 / theta;
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

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

// Tangent of the classical Jacobi rotation that annihilates s_pq:
// tan(2 theta) = 2 s_pq / (s_qq - s_pp), the root of smaller magnitude.
template <typename T>
__device__ __forceinline__ void jacobi_rotation(T app, T aqq, T apq, T& cc, T& ss) {
    const T theta = (aqq - app) / (T(2) * apq);
    T tt;
    if (fabs(theta) > T(1) / num<T>::eps()) tt = T(0.5) / theta;
    else tt = (theta >= T(0) ? T(1) : T(-1)) / (fabs(theta) + sqrt(theta * theta + T(1)));
    cc = T(1) / sqrt(tt * tt + T(1));
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

// Batched block-Jacobi eigensolver for symmetric matrices (float32 / float64).
//
// The SVT of every ALM iteration needs the eigendecomposition of a Gram
// matrix, and the one-time factor needs that of M M^T.  Cyclic block Jacobi
// keeps the work in dense 2b x 2b tiles: in every round the diagonal blocks
// are paired round-robin, each CTA diagonalises one 2b x 2b pivot submatrix
// in shared memory (inner cyclic Jacobi with the classical rotation angle),
// and a second kernel applies the accumulated rotations R_P to the
// off-diagonal tiles (G <- R^T G R) and to the eigenvector matrix (W <- W R).
#include "common.cuh"
#include "inner_jacobi.cuh"
#include "kernels.cuh"

namespace lrr {
namespace {

constexpr int NT = 256;

// threads of a pivot's CTA
template <typename T> __host__ __device__ constexpr int solve_threads() { return sizeof(T) == 8 ? 384 : 1024; }

// global row of local index i (0..2b-1) of the pivot pair (a, c)
__device__ __forceinline__ int pair_row(int i, int a, int c, int b) { return i < b ? a * b + i : c * b + (i - b); }

// Cyclic Jacobi on one pivot in shared memory: B2/2 disjoint rotations per
// round (angle from tan(2 theta) = 2 s_pq / (s_qq - s_pp)), accumulated into R.
// An entry is rotated while |s_pq| > eps sqrt(|s_pp s_qq|) and |s_pq| > floor_rot.
// The fused multiply-adds are written out: which product of a sum of two is
// rounded first is part of the arithmetic the two forms share.

// float32 (64 x 64, one sweep): thread (k, l) of 32 x 32 owns the 2 x 2 sub-block
// of pairs k and l and two rows of R's pair l; it works out pair k's rotation
// itself, takes pair l's from the lane that has it and writes the other S
// buffer, so a round has one barrier.  Bound by shared memory (19 accesses a
// thread and round): 70 us a pivot of the 500 x 500 Gram, 81 with 256 threads
// and a barrier on either side of the rotations.
template <int B2, int LS>
__device__ int inner_sweep_f32(float (*S2)[B2 * LS], float* R, float floor_rot, int* cur_out) {
    constexpr int b = B2 / 2;
    static_assert(b == 32 && solve_threads<float>() == b * b, "a warp holds every pair's rotation");
    const int k = threadIdx.x % b, l = threadIdx.x / b;
    int rotated = 0, cur = 0;
    int p = k, q = B2 - 1 - k, u = l, v = B2 - 1 - l;       // the circle method's round 0
    for (int r = 0; r < B2 - 1; ++r) {
        const float* const S = S2[cur];
        float* const D = S2[cur ^ 1];
        const float app = S[p * LS + p], aqq = S[q * LS + q], apq = S[p * LS + q];
        const float s_pu = S[p * LS + u], s_pv = S[p * LS + v], s_qu = S[q * LS + u], s_qv = S[q * LS + v];
        const float x0 = R[k * LS + u], y0 = R[k * LS + v], x1 = R[(k + b) * LS + u], y1 = R[(k + b) * LS + v];
        const bool act = fabsf(apq) > floor_rot && above_eps_root(fabsf(apq), fabsf(app * aqq));
        float ck, sk;
        jacobi_rotation<float>(app, aqq, apq, ck, sk);
        ck = act ? ck : 1.f;
        sk = act ? sk : 0.f;
        rotated |= act;
        const float cl = __shfl_sync(0xffffffffu, ck, l), sl = __shfl_sync(0xffffffffu, sk, l);
        const float r_pu = fmaf(ck, s_pu, -(sk * s_qu)), r_pv = fmaf(ck, s_pv, -(sk * s_qv));
        const float r_qu = fmaf(sk, s_pu, ck * s_qu), r_qv = fmaf(sk, s_pv, ck * s_qv);
        // the rotated pair's own off-diagonal entries are zero by construction
        const bool own = k == l && sk != 0.f;
        D[p * LS + u] = fmaf(cl, r_pu, -(sl * r_pv));
        D[p * LS + v] = own ? 0.f : fmaf(sl, r_pu, cl * r_pv);
        D[q * LS + u] = own ? 0.f : fmaf(cl, r_qu, -(sl * r_qv));
        D[q * LS + v] = fmaf(sl, r_qu, cl * r_qv);
        R[k * LS + u] = fmaf(cl, x0, -(sl * y0));
        R[k * LS + v] = fmaf(sl, x0, cl * y0);
        R[(k + b) * LS + u] = fmaf(cl, x1, -(sl * y1));
        R[(k + b) * LS + v] = fmaf(sl, x1, cl * y1);
        cur ^= 1;
        p = k ? (p == B2 - 1 ? 1 : p + 1) : 0;
        u = l ? (u == B2 - 1 ? 1 : u + 1) : 0;
        q = q == B2 - 1 ? 1 : q + 1;
        v = v == B2 - 1 ? 1 : v + 1;
        __syncthreads();
    }
    *cur_out = cur;
    return __syncthreads_or(rotated);
}

// log2(|apq| / sqrt|app aqq|) in float32, to 2^-19, from exponents and top
// mantissa bits; false near the ends of the range, where it is not defined.
// (The float64 product, root and compares of the exact form are 800 cycles.)
__device__ __forceinline__ float log2_mantissa(double x) {
    float l;
    const int m = ((__double2hiint(x) & 0x000FFFFF) << 3) | (int)((unsigned)__double2loint(x) >> 29);
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(__int_as_float(0x3F800000 | m)));
    return l;
}
__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ bool log2_ratio(double app, double aqq, double apq, float& d) {
    const int ep = exponent(app), eq = exponent(aqq), eo = exponent(apq);
    const float l = log2_mantissa(apq) - 0.5f * (log2_mantissa(app) + log2_mantissa(aqq));
    d = 0.5f * (float)(2 * eo - ep - eq) + l;
    return ep >= 64 && ep < 1982 && eq >= 64 && eq < 1982 && eo < 1982 && ep + eq >= 1084 && ep + eq <= 3004;
}
__device__ __forceinline__ double negated(double x) {
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
// |x| > y >= 0, x not a NaN (bit patterns order like the values)
__device__ __forceinline__ bool abs_above(double x, double y) {
    return (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll) > __double_as_longlong(y);
}
// |apq| > floor_rot and |apq| > eps sqrt(|app aqq|) in float64, exactly: root and
// product are taken only where the estimate does not decide (entries that are
// rounding noise lie near eps: an estimate to 7 % left one in every few rounds
// undecided)
__device__ __forceinline__ bool must_rotate(double app, double aqq, double apq, double floor_rot) {
    float d;
    if (!abs_above(apq, floor_rot)) return false;
    if (log2_ratio(app, aqq, apq, d) && fabsf(d + 52.f) > 1e-4f) return d > -52.f;
    return fabs(apq) > floor_rot && fabs(apq) > DBL_EPSILON * sqrt(fabs(app * aqq));
}

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// float64 (32 x 32, up to max_sweeps; it stops after a sweep in which no entry
// above floor_sig was rotated).  Bound by the latency of the float64 unit (65
// cycles an operation, one warp instruction every 19 whatever its lanes) along
// the chain from one round's rotations to the next's.  So warp 0 does nothing
// but that chain: it finds the pairs that rotate (6 or 7 of a round's 16, none
// in one round of eight), works out their rotations, lists them for the other
// eight warps and goes on to the next round's diagonal and pair entries on its
// own, from the two-by-two blocks they lie in; the others update the listed
// pairs' rows and columns of S, and R, behind it, and it waits for them only
// before it reads S again.  The schedule moves every pair's item by one
// position a round, so the lanes that hold the two pairs a new pair comes from
// are fixed.  A round takes 3900 cycles, 2100 of them the rotations and 1100 the
// next entries (6400 with every step between barriers of the whole CTA): 204 us
// a pivot of the 500 x 500 Gram, 466 when every 2 x 2 sub-block was updated every
// round.  The warps that share warp 0's scheduler are left out of the updates.
template <int B2, int LS>
__device__ int inner_sweeps_f64(double* S, double* R, double2 (*cs)[B2 / 2], int2 (*pq)[B2 / 2], int* count,
                                double floor_rot, double floor_sig, int max_sweeps) {
    constexpr int b = B2 / 2, NW = 9 * 32, NB = NW + 32;
    static_assert(b == 16, "lanes 16 to 31 repeat lanes 0 to 15");
    const int t = threadIdx.x;
    // barriers: 1 S is up to date (the others arrive, warp 0 waits), 2 a list is
    // out (warp 0 arrives, the others wait), 3 among the others
    if (t < 32) {
        const int k = t & (b - 1);
        const bool first = k == 0, last = k == b - 1, low = t < b;
        int p = circle_item(k, 0, B2), q = circle_item(B2 - 1 - k, 0, B2), any = 0, buf = 0;
        double app = S[p * LS + p], aqq = S[q * LS + q], apq = S[p * LS + q];
        bool pending = false;
        for (int sweep = 0; sweep < max_sweeps; ++sweep) {
            int sig = 0;
            for (int r = 0; r < B2 - 1; ++r) {
                const bool act = must_rotate(app, aqq, apq, floor_rot);
                const unsigned m = __ballot_sync(0xffffffffu, act) & ((1u << b) - 1);
                // the pairs the next round's pair k comes from: A, whose p (k = 15: q)
                // is its p, and B, whose q (k = 0: p) is its q
                const int pd = __shfl_down_sync(0xffffffffu, p, 1, b), qd = __shfl_down_sync(0xffffffffu, q, 1, b);
                const int pu = __shfl_up_sync(0xffffffffu, p, 1, b), qu = __shfl_up_sync(0xffffffffu, q, 1, b);
                const bool own = first || last;
                const int pA = own ? p : pd, qA = own ? q : qd, pB = first ? pd : pu, qB = first ? qd : qu;
                if (!m) {
                    if (pending) bar_sync(1, NB);
                    pending = false;
                    apq = S[(last ? qA : pA) * LS + (first ? pB : qB)];
                } else {
                    any = 1;
                    double c = 1.0, s = 0.0;
                    if (act) jacobi_rotation<double>(app, aqq, apq, c, s);
                    if (pending) bar_sync(1, NB);
                    const double aqp = S[q * LS + p];
                    const double e00 = S[pA * LS + pB], e01 = S[pA * LS + qB];
                    const double e10 = S[qA * LS + pB], e11 = S[qA * LS + qB];
                    if (act && t < b) {
                        const int at = __popc(m & ((1u << k) - 1));
                        cs[buf][at] = make_double2(c, s);
                        pq[buf][at] = make_int2(p, q);
                    }
                    if (t == 0) count[buf] = __popc(m);
                    if (act && abs_above(apq, floor_sig) && abs_above(s, 0.0)) sig = 1;
                    const double cd = __shfl_down_sync(0xffffffffu, c, 1, b), sd = __shfl_down_sync(0xffffffffu, s, 1, b);
                    const double cu = __shfl_up_sync(0xffffffffu, c, 1, b), su = __shfl_up_sync(0xffffffffu, s, 1, b);
                    const double cA = own ? c : cd, sA = own ? s : sd, cB = first ? cd : cu, sB = first ? sd : su;
                    const bool actA = (m >> (own ? k : k + 1)) & 1, actB = (m >> (first ? 1 : k - 1)) & 1;
                    // rows, then columns, as the others do them; the lower lanes take
                    // the p row and the first column, the upper ones the q row and the
                    // second (a float64 operation costs the same for any lanes)
                    const double f = low ? c : s, g = low ? negated(s) : c;
                    const double fA = last ? sA : cA, gA = last ? cA : negated(sA), fB = first ? cB : sB, gB = first ? negated(sB) : cB;
                    const double e0 = low ? e00 : e01, e1 = low ? e10 : e11;
                    const double r0 = fma(f, app, g * aqp), r1 = fma(f, apq, g * aqq);
                    double x = fma(fA, e0, gA * e1);
                    x = actA ? x : last ? e1 : e0;
                    const double y = __shfl_down_sync(0xffffffffu, x, b), d = fma(f, r0, g * r1);
                    const double z = fma(fB, x, gB * y), dq = __shfl_down_sync(0xffffffffu, d, b);
                    apq = __shfl_sync(0xffffffffu, actB ? z : first ? x : y, k);
                    app = __shfl_sync(0xffffffffu, act ? d : app, k);
                    aqq = __shfl_sync(0xffffffffu, act ? dq : aqq, k);
                    bar_arrive(2, NB);
                    pending = true;
                    buf ^= 1;
                }
                const double ad = __shfl_down_sync(0xffffffffu, app, 1, b), au = __shfl_up_sync(0xffffffffu, aqq, 1, b);
                app = first ? app : last ? aqq : ad;
                aqq = first ? ad : au;
                p = last ? qA : pA;
                q = first ? pB : qB;
            }
            if (!__any_sync(0xffffffffu, sig)) break;
        }
        if (pending) bar_sync(1, NB);
        if (t == 0) { count[buf] = -1; count[2] = any; }
        __syncwarp();
        bar_arrive(2, NB);
    } else if (t / 32 % 4 != 0) {
        const int lane = t & 31, w = t / 32 - 1 - t / 128;
        for (int buf = 0;; buf ^= 1) {
            bar_sync(2, NB);
            const int n = count[buf];
            if (n < 0) break;
            // rows p and q of every rotating pair
            for (int i = w; i < n; i += NW / 32) {
                const int2 v = pq[buf][i];
                const double2 r2 = cs[buf][i];
                double* const A = S + lane;
                const double x = A[v.x * LS], y = A[v.y * LS];
                A[v.x * LS] = fma(r2.x, x, -(r2.y * y));
                A[v.y * LS] = fma(r2.y, x, r2.x * y);
            }
            bar_sync(3, NW);
            // columns; the pair's own off-diagonal entries are zero by construction
            for (int i = w; i < n; i += NW / 32) {
                const int2 v = pq[buf][i];
                const double2 r2 = cs[buf][i];
                double* const A = S + lane * LS;
                const double x = A[v.x], y = A[v.y];
                A[v.x] = lane == v.y && r2.y != 0.0 ? 0.0 : fma(r2.x, x, -(r2.y * y));
                A[v.y] = lane == v.x && r2.y != 0.0 ? 0.0 : fma(r2.y, x, r2.x * y);
            }
            bar_arrive(1, NB);
            for (int i = w; i < n; i += NW / 32) {
                const int2 v = pq[buf][i];
                const double2 r2 = cs[buf][i];
                double* const A = R + lane * LS;
                const double x = A[v.x], y = A[v.y];
                A[v.x] = fma(r2.x, x, -(r2.y * y));
                A[v.y] = fma(r2.y, x, r2.x * y);
            }
        }
    }
    __syncthreads();
    return count[2];
}

template <typename T, int B2>
__global__ void __launch_bounds__(solve_threads<T>()) jac_solve(const JacDesc<T>* __restrict__ descs, int round, T tol) {
    constexpr int b = B2 / 2, NS = solve_threads<T>(), LS = sizeof(T) == 8 ? B2 + 1 : B2 + 2;
    const JacDesc<T> d = descs[blockIdx.y];
    if (d.active && *d.active == 0) return;
    if (*d.done) return;
    const int nb = d.pp / b, npairs = nb / 2;
    const int P = blockIdx.x;
    if (P >= npairs) return;
    const int a = circle_item(P, round, nb), c = circle_item(nb - 1 - P, round, nb);

    extern __shared__ __align__(16) unsigned char jac_smem[];
    T* const S0 = reinterpret_cast<T*>(jac_smem);            // float32: two buffers
    T* const R = S0 + (sizeof(T) == 8 ? 1 : 2) * B2 * LS;
    __shared__ double2 cs[2][b];
    __shared__ int2 pq[2][b];
    __shared__ int count[3];
    __shared__ T red[NS / 32];
    const int t = threadIdx.x;
    // Off-diagonal entries below the rounding noise of the Gram products
    // (~sqrt(order) * eps * max|G_ii|) carry no information and do not count
    // towards the convergence measure; they are still rotated away like any
    // other entry above eps * sqrt(G_ii G_jj), so a converged sweep leaves the
    // resolved part of the spectrum at working accuracy.
    const T floor_abs = T(4) * sqrt(T(d.pp)) * num<T>::eps() * (*d.scale) + num<T>::tiny();
    const T floor_rot = num<T>::eps() * num<T>::eps() * (*d.scale) + num<T>::tiny();

    for (int e = t; e < B2 * B2; e += NS) {
        const int i = e % B2, j = e / B2;
        S0[i * LS + j] = d.G[pair_row(i, a, c, b) + (int64_t)pair_row(j, a, c, b) * d.pp];
        R[i * LS + j] = (i == j) ? T(1) : T(0);
    }
    __syncthreads();

    // convergence measure of this pivot block before rotating it, and whether
    // any entry is large enough to rotate at all
    T offm = T(0);
    int any = 0;
    const float log2_tol = log2f((float)tol);
    for (int e = t; e < B2 * B2; e += NS) {
        const int i = e % B2, j = e / B2;
        if (i < j) {
            const T v = fabs(S0[i * LS + j]);
            if constexpr (sizeof(T) == 8) {
                // only the comparison with tol is used of the measure
                float d;
                any |= must_rotate(S0[i * LS + i], S0[j * LS + j], v, floor_rot);
                if (!abs_above(v, floor_abs)) continue;
                if (log2_ratio(S0[i * LS + i], S0[j * LS + j], v, d) && fabsf(d - log2_tol) > 1e-3f) {
                    if (d > log2_tol) offm = T(2) * tol;
                    continue;
                }
            }
            const T sc = sqrt(fabs(S0[i * LS + i] * S0[j * LS + j]));
            if (v > floor_abs) offm = fmax(offm, v / (sc + num<T>::tiny()));
            if (sizeof(T) == 4 && v > floor_rot && v > num<T>::eps() * sc) any = 1;
        }
    }
    offm = warp_max(offm);
    if ((t & 31) == 0) red[t >> 5] = offm;
    __syncthreads();
    if (t == 0) {
        T mx = T(0);
        for (int w = 0; w < NS / 32; ++w) mx = fmax(mx, red[w]);
        atomic_max_nonneg(d.off, mx);
    }
    const bool need = __syncthreads_or(any) != 0;

    // float32 (the start of the setup's eigendecomposition): one inner sweep
    // per pivot, the outer sweeps continue from there; float64: up to six
    int any_rot = 0, cur = 0;
    if (need) {
        if constexpr (sizeof(T) == 8) any_rot = inner_sweeps_f64<B2, LS>(S0, R, cs, pq, count, floor_rot, floor_abs, 6);
        else any_rot = inner_sweep_f32<B2, LS>(reinterpret_cast<float(*)[B2 * LS]>(S0), R, floor_rot, &cur);
    }
    // diagonalised pivot block back into G, rotation out for the apply kernel
    if (t == 0) d.rot[P] = any_rot;
    if (any_rot) {
        const T* const S = S0 + cur * B2 * LS;
        T* Rg = d.R + (int64_t)P * B2 * B2;
        for (int e = t; e < B2 * B2; e += NS) {
            const int i = e % B2, j = e / B2;
            d.G[pair_row(i, a, c, b) + (int64_t)pair_row(j, a, c, b) * d.pp] = S[i * LS + j];
            Rg[e] = R[i * LS + j];
        }
    }
}

template <typename T, int B2>
__global__ void __launch_bounds__(NT) jac_apply(const JacDesc<T>* __restrict__ descs, int round) {
    constexpr int b = B2 / 2;
    const JacDesc<T> d = descs[blockIdx.y];
    if (d.active && *d.active == 0) return;
    if (*d.done) return;
    const int nb = d.pp / b, npairs = nb / 2;
    const int ntile_g = npairs * (npairs - 1) / 2;
    int tile = blockIdx.x;
    if (tile >= ntile_g + npairs * npairs) return;

    __shared__ T X[B2][B2 + 1];
    __shared__ T Q[B2][B2 + 1];
    const int t = threadIdx.x;
    // each thread owns 16 (B2=64) or 4 (B2=32) output entries: rows i0 + 16*ii, cols tj
    constexpr int PER = B2 * B2 / NT;

    if (tile < ntile_g) {
        // off-diagonal tile (P, Q), P < Q:  G[I_P, I_Q] <- R_P^T G[I_P, I_Q] R_Q
        int P = 0, rem = tile;
        while (rem >= npairs - 1 - P) { rem -= npairs - 1 - P; ++P; }
        const int Qp = P + 1 + rem;
        const int rP = d.rot[P], rQ = d.rot[Qp];
        if (!rP && !rQ) return;
        const int a = circle_item(P, round, nb), c = circle_item(nb - 1 - P, round, nb);
        const int a2 = circle_item(Qp, round, nb), c2 = circle_item(nb - 1 - Qp, round, nb);
        const T* RP = d.R + (int64_t)P * B2 * B2;
        const T* RQ = d.R + (int64_t)Qp * B2 * B2;
        for (int e = t; e < B2 * B2; e += NT) {
            const int i = e % B2, j = e / B2;
            X[i][j] = d.G[pair_row(i, a, c, b) + (int64_t)pair_row(j, a2, c2, b) * d.pp];
            Q[i][j] = rQ ? RQ[e] : (i == j ? T(1) : T(0));
        }
        __syncthreads();
        T acc[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int e = t + u * NT, i = e % B2, j = e / B2;
            T s = T(0);
#pragma unroll 8
            for (int k = 0; k < B2; ++k) s = fma(X[i][k], Q[k][j], s);
            acc[u] = s;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int e = t + u * NT, i = e % B2, j = e / B2;
            X[i][j] = acc[u];
            Q[i][j] = rP ? RP[e] : (i == j ? T(1) : T(0));
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int e = t + u * NT, i = e % B2, j = e / B2;
            T s = T(0);
#pragma unroll 8
            for (int k = 0; k < B2; ++k) s = fma(Q[k][i], X[k][j], s);
            const int gi = pair_row(i, a, c, b), gj = pair_row(j, a2, c2, b);
            d.G[gi + (int64_t)gj * d.pp] = s;
            d.G[gj + (int64_t)gi * d.pp] = s;
        }
    } else {
        // eigenvector tile: rows chunk ch, columns I_P:  W[ch, I_P] <- W[ch, I_P] R_P
        tile -= ntile_g;
        const int P = tile % npairs, ch = tile / npairs;
        if (!d.rot[P]) return;
        const int a = circle_item(P, round, nb), c = circle_item(nb - 1 - P, round, nb);
        const T* RP = d.R + (int64_t)P * B2 * B2;
        for (int e = t; e < B2 * B2; e += NT) {
            const int i = e % B2, j = e / B2;
            X[i][j] = d.W[(ch * B2 + i) + (int64_t)pair_row(j, a, c, b) * d.pp];
            Q[i][j] = RP[e];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int e = t + u * NT, i = e % B2, j = e / B2;
            T s = T(0);
#pragma unroll 8
            for (int k = 0; k < B2; ++k) s = fma(X[i][k], Q[k][j], s);
            d.W[(ch * B2 + i) + (int64_t)pair_row(j, a, c, b) * d.pp] = s;
        }
    }
}

template <typename T>
__global__ void jac_reset(const JacDesc<T>* __restrict__ descs, int nmat) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nmat) return;
    *descs[i].done = 0;
    *descs[i].off = T(0);
}

template <typename T>
__global__ void jac_check(const JacDesc<T>* __restrict__ descs, int nmat, T tol) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nmat) return;
    const JacDesc<T> d = descs[i];
    if (*d.done == 0 && *d.off <= tol) *d.done = 1;
    *d.off = T(0);
}

}  // namespace

template <typename T>
cudaError_t jacobi_sweeps(const JacDesc<T>* d_desc, int nmat, int max_pp, int sweeps, T tol, cudaStream_t s,
                         const int* done_dev, int* sweeps_run) {
    constexpr int b = jacobi_bs<T>();
    constexpr int B2 = 2 * b;
    if (sweeps_run) *sweeps_run = 0;
    if (nmat <= 0 || max_pp <= 0) return cudaSuccess;
    const int nb = max_pp / b, npairs = nb / 2;
    jac_reset<T><<<ceil_div(nmat, 128), 128, 0, s>>>(d_desc, nmat);
    const dim3 gs((unsigned)npairs, (unsigned)nmat);
    constexpr int LS = sizeof(T) == 8 ? B2 + 1 : B2 + 2;
    constexpr int smem = (int)sizeof(T) * B2 * LS * (sizeof(T) == 8 ? 2 : 3);      // S (float32: twice) and R
    static std::atomic<uint64_t> smem_set{0};
    const cudaError_t ea = ensure_smem_limit(jac_solve<T, B2>, smem, smem_set);
    if (ea != cudaSuccess) return ea;
    const dim3 ga((unsigned)(npairs * (npairs - 1) / 2 + npairs * npairs), (unsigned)nmat);
    for (int sw = 0; sw < sweeps; ++sw) {
        for (int r = 0; r < nb - 1; ++r) {
            jac_solve<T, B2><<<gs, solve_threads<T>(), smem, s>>>(d_desc, r, tol);
            jac_apply<T, B2><<<ga, NT, 0, s>>>(d_desc, r);
        }
        jac_check<T><<<ceil_div(nmat, 128), 128, 0, s>>>(d_desc, nmat, tol);
        if (sweeps_run) *sweeps_run = sw + 1;
        if (done_dev) {
            // one matrix: stop launching once it has converged
            int done = 0;
            cudaError_t e = cudaMemcpyAsync(&done, done_dev, sizeof(int), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return e;
            if (done) break;
        }
    }
    return cudaGetLastError();
}

template cudaError_t jacobi_sweeps<float>(const JacDesc<float>*, int, int, int, float, cudaStream_t, const int*,
                                          int*);
template cudaError_t jacobi_sweeps<double>(const JacDesc<double>*, int, int, int, double, cudaStream_t, const int*,
                                           int*);

}  // namespace lrr

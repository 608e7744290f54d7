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
template <typename T> __host__ __device__ constexpr int solve_threads() { return sizeof(T) == 8 ? 256 : 1024; }

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
// buffer, so a round has one barrier (0.3 us; 1.3 us with 256 threads and a
// barrier on either side of the rotations: 81 us a pivot, now 20).
template <int B2, int LS>
__device__ int inner_sweep_f32(float (*S2)[B2 * LS], float* R, float floor_rot, int* cur_out) {
    constexpr int b = B2 / 2;
    static_assert(b == 32 && solve_threads<float>() == b * b, "a warp holds every pair's rotation");
    const int k = threadIdx.x % b, l = threadIdx.x / b;
    int rotated = 0, cur = 0;
    for (int r = 0; r < B2 - 1; ++r) {
        const int p = circle_item(k, r, B2), q = circle_item(B2 - 1 - k, r, B2);
        const int u = circle_item(l, r, B2), v = circle_item(B2 - 1 - l, r, B2);
        const float* const S = S2[cur];
        float* const D = S2[cur ^ 1];
        const float app = S[p * LS + p], aqq = S[q * LS + q], apq = S[p * LS + q];
        const float s_pu = S[p * LS + u], s_pv = S[p * LS + v], s_qu = S[q * LS + u], s_qv = S[q * LS + v];
        const float x0 = R[k * LS + u], y0 = R[k * LS + v], x1 = R[(k + b) * LS + u], y1 = R[(k + b) * LS + v];
        const bool act = fabsf(apq) > floor_rot && fabsf(apq) > FLT_EPSILON * sqrtf(fabsf(app * aqq));
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
        __syncthreads();
    }
    *cur_out = cur;
    return __syncthreads_or(rotated);
}

// |apq| > eps sqrt(|app aqq|) in float64, exactly; the square root is taken only
// where an estimate from the exponent (0 to 6.1 % above it) does not decide
__device__ __forceinline__ bool above_eps(double app, double aqq, double apq) {
    const double g = fabs(app * aqq);
    const double est = __hiloint2double((__double2hiint(g) >> 1) + 0x1FF80000, 0);
    if (g > 1e-290) {
        if (apq > 1.001 * DBL_EPSILON * est) return true;
        if (apq < 0.94 * DBL_EPSILON * est) return false;
    }
    return apq > DBL_EPSILON * sqrt(g);
}

// float64 (32 x 32, up to max_sweeps; it stops after a sweep in which no entry
// above floor_sig was rotated).  Bound by the float64 units (two FMA lanes per SM
// and clock) and their latency, and on average only 5 or 6 of a round's 16 pairs
// still rotate: so a round first finds those, and only their rows, then their
// columns, are touched; an idle round ends at its first barrier.  (Every 2 x 2
// sub-block every round: 466 us a pivot on the 500 x 5000 problem, now 360, of
// which the rotations themselves, a chain of three divisions and two square roots,
// are 60 %.)
template <int B2, int LS>
__device__ int inner_sweeps_f64(double* S, double* R, double2* cs, int2* pq, int* count2, double floor_rot,
                                double floor_sig, int max_sweeps) {
    constexpr int b = B2 / 2;
    const int t = threadIdx.x;
    int any = 0, phase = 0;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        int sig = 0;
        for (int r = 0; r < B2 - 1; ++r, phase ^= 1) {
            if (t < 32) {
                bool act = false;
                double c = 1.0, sv = 0.0;
                const int k = t & (b - 1);
                const int p = circle_item(k, r, B2), q = circle_item(B2 - 1 - k, r, B2);
                if (t < b) {
                    const double app = S[p * LS + p], aqq = S[q * LS + q], apq = S[p * LS + q];
                    act = fabs(apq) > floor_rot && above_eps(app, aqq, fabs(apq));
                    if (act) {
                        jacobi_rotation<double>(app, aqq, apq, c, sv);
                        if (fabs(apq) > floor_sig && fabs(sv) > 0.0) sig = 1;
                    }
                }
                // the rotating pairs, listed
                const unsigned m = __ballot_sync(0xffffffffu, act);
                if (act) {
                    const int at = __popc(m & ((1u << t) - 1));
                    cs[at] = make_double2(c, sv);
                    pq[at] = make_int2(p, q);
                }
                if (t == 0) count2[phase] = __popc(m);
            }
            __syncthreads();
            const int cnt = count2[phase] * B2;
            if (!cnt) continue;
            any = 1;
            // rows p and q of every rotating pair
            for (int e = t; e < cnt; e += NT) {
                const int j = e % B2;
                const int2 w = pq[e / B2];
                const double2 r2 = cs[e / B2];
                const double x = S[w.x * LS + j], y = S[w.y * LS + j];
                S[w.x * LS + j] = fma(r2.x, x, -(r2.y * y));
                S[w.y * LS + j] = fma(r2.y, x, r2.x * y);
            }
            __syncthreads();
            // columns, and R
            for (int e = t; e < 2 * cnt; e += NT) {
                const bool isr = e >= cnt;
                const int f = isr ? e - cnt : e, i = f % B2;
                const int2 w = pq[f / B2];
                const double2 r2 = cs[f / B2];
                double* const A = (isr ? R : S) + i * LS;
                const double x = A[w.x], y = A[w.y];
                // the pair's own off-diagonal entries are zero by construction
                A[w.x] = !isr && i == w.y && r2.y != 0.0 ? 0.0 : fma(r2.x, x, -(r2.y * y));
                A[w.y] = !isr && i == w.x && r2.y != 0.0 ? 0.0 : fma(r2.y, x, r2.x * y);
            }
            __syncthreads();
        }
        if (!__syncthreads_or(sig)) break;
    }
    return any;
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
    __shared__ double2 cs[b];
    __shared__ int2 pq[b];
    __shared__ int count2[2];
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
    for (int e = t; e < B2 * B2; e += NS) {
        const int i = e % B2, j = e / B2;
        if (i < j) {
            const T v = fabs(S0[i * LS + j]);
            const T sc = sqrt(fabs(S0[i * LS + i] * S0[j * LS + j]));
            if (v > floor_abs) offm = fmax(offm, v / (sc + num<T>::tiny()));
            if (v > floor_rot && v > num<T>::eps() * sc) any = 1;
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
        if constexpr (sizeof(T) == 8) any_rot = inner_sweeps_f64<B2, LS>(S0, R, cs, pq, count2, floor_rot, floor_abs, 6);
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

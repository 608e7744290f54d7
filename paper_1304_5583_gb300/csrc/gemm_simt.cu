// Grouped general matrix product on the CUDA cores (float32 / float64).
// This is the accurate product of the plain-precision path: every group is an
// independent column-major product C = alpha op(A) op(B) + beta C.
//
// Every element is the sum of 16-term slabs: a slab's products run in a fresh
// partial, which is then added to the element's total.  (One long chain of FMAs
// into a single register lets rounding grow with K; with K in the thousands it
// doubled the float32 error of the iterate on face-like data.)  Neither the
// tile nor the staging touches that order, so they change no bit of C.
//
// 128 threads to a tile, TM x TN elements each, K slabs of 16 brought to shared
// memory by cp.async in a ring of four (a slab's loads take about as long as two
// slabs' products at the solver's sizes; with one buffer and two barriers a
// slab they were waited for in full).  A warp's lanes lie 8 along N and 4 along
// M: the 16-byte reads of A are then uniform over eight lanes, and per 32 FMAs a
// lane makes three reads that take the shared memory as long as the FMAs take
// the FMA units (64 x 64 tiles; eight scalar reads per 16 FMAs took twice that).
// C leaves through shared memory so that stores run along its columns.
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace lrr {
namespace {

constexpr int NT = 128, BK = 16, STAGES = 4;

template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = ok ? BYTES : 0;      // 0: zero fill
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES), "r"(n));
}

// N consecutive values from shared memory, 16 bytes at a time where they fill that
template <typename T, int N>
__device__ __forceinline__ void read_row(const T* p, T (&v)[N]) {
    constexpr int V = 16 / sizeof(T);
    if constexpr (N % V == 0) {
#pragma unroll
        for (int i = 0; i < N; i += V) {
            const uint4 q = *reinterpret_cast<const uint4*>(p + i);
            const T* const w = reinterpret_cast<const T*>(&q);
#pragma unroll
            for (int e = 0; e < V; ++e) v[i + e] = w[e];
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = p[i];
    }
}

// One operand's slab, rows i of the tile (BX of them) by 16 k: K runs along
// memory when TR, the tile's rows otherwise.  Element (i, kk) lands at
// S[kk * LD + i]; out of range is zero.
template <typename T, bool TR, int BX, int LD>
__device__ __forceinline__ void load_slab(T* S, const T* P, int64_t ld, int x0, int X, int k0, int K, bool vec) {
    const int t = threadIdx.x;
    if constexpr (TR) {
        const int kk = t % BK;
        const bool kok = k0 + kk < K;
#pragma unroll
        for (int i = t / BK; i < BX; i += NT / BK) {
            const bool ok = kok && x0 + i < X;
            copy_async<sizeof(T)>(S + kk * LD + i, ok ? P + k0 + kk + (int64_t)(x0 + i) * ld : P, ok);
        }
    } else {
        constexpr int V = 16 / sizeof(T);
        if (vec) {          // 16-byte aligned columns; the last rows may be partial
            constexpr int Q = BX / V;
#pragma unroll
            for (int e = t; e < BK * Q; e += NT) {
                const int i = e % Q * V, kk = e / Q;
                const int left = k0 + kk < K ? X - (x0 + i) : 0;
                const T* const src = P + x0 + i + (int64_t)(k0 + kk) * ld;
                const unsigned d = (unsigned)__cvta_generic_to_shared(S + kk * LD + i);
                const int n = left >= V ? 16 : left > 0 ? left * (int)sizeof(T) : 0;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(n ? src : P), "r"(n));
            }
        } else {
#pragma unroll
            for (int e = t; e < BK * BX; e += NT) {
                const int i = e % BX, kk = e / BX;
                const bool ok = x0 + i < X && k0 + kk < K;
                copy_async<sizeof(T)>(S + kk * LD + i, ok ? P + x0 + i + (int64_t)(k0 + kk) * ld : P, ok);
            }
        }
    }
}

// CTAs to an SM the registers are cut for: four of the float32 64 x 64 tiles (128
// registers: M Z of the 600 x 6000 solve 88 -> 75 us), but three when both
// operands run along K (U^T P: 90 us at three, 118 at four, where it spills).
template <typename T, bool TA, bool TB, int TM>
constexpr int min_ctas() { return sizeof(T) == 4 && TM == 8 ? (TA && !TB ? 3 : 4) : 1; }

template <typename T, bool TA, bool TB, int TM, int TN>
__global__ void __launch_bounds__(NT, min_ctas<T, TA, TB, TM>()) gemm_kernel(const GemmDesc<T>* __restrict__ descs, int tiles_m) {
    constexpr int BM = 8 * TM, BN = 16 * TN, V = 16 / sizeof(T);
    constexpr int LA = BM + V, LB = BN + V, SLAB = BK * (LA + LB);
    static_assert(BN * LA <= STAGES * SLAB, "C leaves through the ring");
    const GemmDesc<T> d = descs[blockIdx.z];
    if (d.flag && *d.flag == 0) return;
    const int tm = blockIdx.x % tiles_m, tn = blockIdx.x / tiles_m;
    const int m0 = tm * BM, n0 = tn * BN;
    if (m0 >= d.m || n0 >= d.n) return;
    // A^T A and A A^T: the tiles above the diagonal are computed and stored twice
    // (the mirrored element has the same products in the same order)
    static_assert(BM == BN, "square tiles");
    const bool sym = TA != TB && d.A == d.B && d.lda == d.ldb && d.m == d.n && d.beta == T(0) && !d.ccol && !d.kscale &&
                     !d.absmax;
    if (sym && tm > tn) return;

    extern __shared__ __align__(16) unsigned char gemm_smem[];
    T* const ring = reinterpret_cast<T*>(gemm_smem);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int wm = (warp & 1) * (BM / 2) + (lane >> 3) * TM, wn = (warp >> 1) * (BN / 2) + (lane & 7) * TN;
    const bool va = reinterpret_cast<uintptr_t>(d.A) % 16 == 0 && d.lda % V == 0;
    const bool vb = reinterpret_cast<uintptr_t>(d.B) % 16 == 0 && d.ldb % V == 0;
    const int nk = (d.k + BK - 1) / BK;

    // A's rows are M: along memory unless TA; B's are N: along memory if TB
    auto fetch = [&](int s) {
        if (s < nk) {
            T* const S = ring + (s % STAGES) * SLAB;
            load_slab<T, TA, BM, LA>(S, d.A, d.lda, m0, d.m, s * BK, d.k, va);
            load_slab<T, !TB, BN, LB>(S + BK * LA, d.B, d.ldb, n0, d.n, s * BK, d.k, vb);
        }
        asm volatile("cp.async.commit_group;\n");
    };
#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) fetch(s);

    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
    for (int s = 0; s < nk; ++s) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(STAGES - 2));
        T* const S = ring + (s % STAGES) * SLAB;
        __syncthreads();          // slab s has landed for all; slab s - 1 is free
        fetch(s + STAGES - 1);
        if (d.kscale) {           // rows of the slab scaled in place (k in each row's order)
            for (int e = t; e < BK * BM; e += NT) {
                const int kk = e / BM, gk = s * BK + kk;
                if (gk < d.k) S[kk * LA + e % BM] *= d.kscale[gk];
            }
            __syncthreads();
        }
        T part[TM][TN];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) part[i][j] = T(0);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[TM], b[TN];
            read_row<T, TM>(S + kk * LA + wm, a);
            read_row<T, TN>(S + BK * LA + kk * LB + wn, b);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) part[i][j] = fma(a[i], b[j], part[i][j]);
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] += part[i][j];
    }
    asm volatile("cp.async.wait_group 0;\n");
    if (d.absmax) {
        T mx = T(0);
#pragma unroll
        for (int j = 0; j < TN; ++j)
#pragma unroll
            for (int i = 0; i < TM; ++i)
                if (n0 + wn + j < d.n && m0 + wm + i < d.m) mx = fmax(mx, fabs(d.alpha * acc[i][j]));
        mx = warp_max(mx);
        if (lane == 0) atomic_max_nonneg(d.absmax, mx);
        return;
    }
    __syncthreads();
    T* const Cs = ring;           // column j of the tile at Cs + j * LA
#pragma unroll
    for (int j = 0; j < TN; ++j)
#pragma unroll
        for (int i = 0; i < TM; ++i) Cs[(wn + j) * LA + wm + i] = d.alpha * acc[i][j];
    __syncthreads();
    for (int e = t; e < BM * BN; e += NT) {
        const int i = e % BM, j = e / BM, gi = m0 + i, gj = n0 + j;
        if (gi >= d.m || gj >= d.n) continue;
        T* const c = d.C + gi + (d.ccol ? d.ccol[gj] : gj) * d.ldc;
        T v = Cs[j * LA + i];
        if (d.beta != T(0)) v = fma(d.beta, *c, v);
        *c = v;
    }
    if (sym && tm != tn)
        for (int e = t; e < BM * BN; e += NT) {
            const int j = e % BN, i = e / BN, gi = m0 + i, gj = n0 + j;
            if (gi < d.m && gj < d.n) d.C[gj + (int64_t)gi * d.ldc] = Cs[j * LA + i];
        }
}

template <typename T, int TM, int TN>
cudaError_t launch(const GemmDesc<T>* d_desc, int groups, bool transA, bool transB, int max_m, int max_n,
                   cudaStream_t s) {
    constexpr int BM = 8 * TM, BN = 16 * TN, V = 16 / sizeof(T);
    constexpr size_t smem = sizeof(T) * STAGES * BK * (BM + BN + 2 * V);
    static_assert(smem <= 48 * 1024 || sizeof(T) == 8, "within the default limit");
    const int tiles_m = (int)ceil_div(max_m, BM), tiles_n = (int)ceil_div(max_n, BN);
    const dim3 grid((unsigned)(tiles_m * tiles_n), 1, (unsigned)groups);
    auto go = [&](auto kernel, std::atomic<uint64_t>& done) {
        const cudaError_t e = ensure_smem_limit(kernel, (int)smem, done);
        if (e != cudaSuccess) return e;
        kernel<<<grid, NT, smem, s>>>(d_desc, tiles_m);
        return cudaGetLastError();
    };
    static std::atomic<uint64_t> set[4];
    if (!transA && !transB) return go(gemm_kernel<T, false, false, TM, TN>, set[0]);
    if (transA && !transB) return go(gemm_kernel<T, true, false, TM, TN>, set[1]);
    if (!transA && transB) return go(gemm_kernel<T, false, true, TM, TN>, set[2]);
    return go(gemm_kernel<T, true, true, TM, TN>, set[3]);
}

}  // namespace

template <typename T>
cudaError_t gemm_grouped(const GemmDesc<T>* d_desc, int groups, bool transA, bool transB, int max_m, int max_n,
                         cudaStream_t s) {
    if (groups <= 0 || max_m <= 0 || max_n <= 0) return cudaSuccess;
    // 64 x 64 tiles where they give every SM one, else 32 x 32 (float64 also
    // 16 x 16): a tile's time is its K loop, so idle SMs are worth the extra
    // operand reads.  float64 is bound by two FMA lanes per SM: 16 tiles of the
    // 100 x 500 x 100 product took 100 us on 16 SMs.
    const int64_t t64 = (int64_t)ceil_div(max_m, 64) * ceil_div(max_n, 64) * groups;
    const int64_t t32 = (int64_t)ceil_div(max_m, 32) * ceil_div(max_n, 32) * groups;
    if (t64 >= 152) return launch<T, 8, 4>(d_desc, groups, transA, transB, max_m, max_n, s);
    if (sizeof(T) == 4 || t32 >= 152) return launch<T, 4, 2>(d_desc, groups, transA, transB, max_m, max_n, s);
    return launch<T, 2, 1>(d_desc, groups, transA, transB, max_m, max_n, s);
}

template cudaError_t gemm_grouped<float>(const GemmDesc<float>*, int, bool, bool, int, int, cudaStream_t);
template cudaError_t gemm_grouped<double>(const GemmDesc<double>*, int, bool, bool, int, int, cudaStream_t);

}  // namespace lrr

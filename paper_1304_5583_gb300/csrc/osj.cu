// Batched one-sided block-Jacobi SVD for the singular-value thresholding step.
//
// For every block the L x p matrix X (X = A W for a tall A, X = A^T W for a
// wide one, W the previous iteration's right basis) is driven to orthogonal
// columns by rotations X <- X R, W <- W R.  The columns are cut into column
// blocks of b; in each round the column blocks are paired round-robin (circle
// method) and every pair (a pivot of 2b columns)
//   1. forms the 2b x 2b Gram S = X_P^T X_P afresh from the columns of X
//      (each entry carries only the rounding of its own two columns),
//   2. rotates S towards diagonal form in shared memory,
//   3. re-orthonormalises the accumulated rotation R and applies it to X_P
//      and W_P in update form.
// Pairs of a round touch disjoint columns.
//
// Two schedules (OsjMode):
//   kept     columns in their own places, one inner pass over all pairs of a
//            pivot.  The float32 solver: its stop test (1e-6 against float32
//            residuals) and the blocks' paths react to the rounding of every
//            SVT, so a pivot's arithmetic is held fixed, operation for operation
//            (which pivots are formed follows from the columns' norms, with
//            margins; see the list of pivots in osj_svd).
//   sorted   columns taken by falling norm (sorted at the start of sweeps 0, 2
//            and 4), up to two inner passes over the pairs that cross the two
//            column blocks (the first round of a sweep also takes the pairs
//            inside each).  The stand-alone SVT and float64.  Small columns
//            come together, so whole pivots need nothing, and sweeps are
//            saved: a cold 350 x 256 float32 SVT that keeps 100 directions
//            takes 9 sweeps and 716 rotated pivots, against 13 and 1262.
//            (Sorting at every sweep shuffles columns of nearly equal norm and
//            slows the float64 tail: 23 sweeps against 12.)
//
// One launch runs every sweep of every block: each block is a thread-block
// cluster whose CTAs share the pivots of a round and meet at a cluster barrier
// between rounds (the barrier's release/acquire makes one round's column
// updates visible to the next).  Where a cluster has more CTAs than a round
// has pivots, `split` CTAs share one pivot: each forms the Gram of its rows,
// the partial Grams meet through distributed shared memory, every member runs
// the same (tiny) inner rotation and applies it to its own rows.  A cluster ends
// at 16 CTAs; the clusterless form (below, `meet`) splits the pivots of a few
// blocks over more of the chip, its CTAs meeting through memory.  A Gram is
// always the sum of the same row-slot partials in the same order, so neither
// the cluster size nor the split nor the form changes a bit of the result.
// After each sweep the cluster reduces the largest convergence measure seen in
// it and stops once that is below the tolerance, so a converged block costs
// nothing further and the others are not held to a common sweep count.
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "common.cuh"
#include "inner_jacobi.cuh"
#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace lrr {
namespace {

// Threads per CTA (a CTA works on one pivot, or one member's share of it, at a
// time).  512, one CTA to an SM, with the pivot's columns of X kept in shared
// memory from the Gram to the rotation, when the blocks' CTAs have the SMs to
// themselves: a pivot's own chain of loads, products and rotations is then all
// there is to wait for (a rotated pivot of the 350 x 256 float32 SVT: 20 us, 8 of
// them the inner rotations, 6 the update, 2 the Gram).  256 at up to 80
// registers, three CTAs to an SM, when there are more blocks than that (or
// columns too long to keep): their phases cover one another's latencies.
constexpr int NT_MANY = 256, NT_FEW = 512;
// A Gram is summed in row slots: of every chunk of 64 rows, slot s has the SR
// rows from SR s (float32: 4 slots of 16 rows, each chunk's 16 products summed on
// their own and then added to the slot's total; float64: 16 of 4).  The slots'
// totals are added in slot order.
constexpr int CHR = 64;
constexpr size_t SMEM_MAX = 227 * 1024;

// Column-block width: float32 16 (pivots of 32 columns).  float64 8: the inner
// rotation is bound by the float64 units (two FMA lanes per SM and clock), and
// a 16-column pivot has an eighth of a 32-column pivot's inner work while a
// round then has twice as many pivots to spread over the SMs.
template <typename T> struct Cfg;
template <> struct Cfg<float> { static constexpr int OB = 16, V = 4, LS = 34, NSLOT = 4, SR = 16; };
template <> struct Cfg<double> { static constexpr int OB = 8, V = 2, LS = 18, NSLOT = 16, SR = 4; };

template <typename T>
struct __align__(16) Smem {                       // followed by the stage
    static constexpr int B2 = 2 * Cfg<T>::OB;
    static constexpr int ST = CHR + Cfg<T>::V;    // column stride of a staged chunk (conflict-free 16-byte reads)
    static constexpr int PS = B2 + Cfg<T>::V;     // row stride of a partial Gram
    static constexpr int PART = Cfg<T>::NSLOT * B2 * PS;  // the partial Grams
    static constexpr int STAGE = PART + 2 * B2 * ST;
    T S[2][B2 * Cfg<T>::LS];
    T R[B2 * Cfg<T>::LS];
    T G[B2 * B2];                                 // R^T R
    T R4[B2 * B2];                                // R - I, rows of 16-byte multiples
    T red[NT_FEW / 32];
    int cid[B2];                                  // physical column of each pivot column, -1: none
    int sig[2], rot, cur, fail;
    OsjDesc<T> d;                                 // the block's descriptor (kept out of the registers)
};

// Shared memory after Smem: the partial Grams; then, with 256 threads, two
// staged chunks, and with 512 the member's rows of the pivot columns of X, and
// of W (at most WROWS of them at a time).  W takes the place of the partial
// Grams, which are read before it is written; a split pivot's partial Grams
// are also read by the other members, so there W has a place of its own.
constexpr int WROWS = 512;
// rows of X of a split pivot's member: of every chunk the NSLOT / split slots it owns
template <typename T>
__host__ __device__ constexpr int local_rows(int L, int split) {
    return (L + CHR - 1) / CHR * (Cfg<T>::NSLOT / split) * Cfg<T>::SR;
}
// column strides of the kept columns: one bank quad past a multiple of 32 words
template <typename T>
__host__ __device__ constexpr int panel_stride(int L, int split) {
    return (local_rows<T>(L, split) + 31) / 32 * 32 + Cfg<T>::V;
}
template <typename T>
__host__ __device__ constexpr int wpanel_stride(int p, int split) {
    const int r = ((p + 31) / 32 + split - 1) / split * 32;
    return (r < WROWS ? r : WROWS) + Cfg<T>::V;
}

// 16-byte vectors of shared memory
__device__ __forceinline__ void lds16(const float* p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void lds16(const double* p, double (&v)[2]) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    v[0] = x.x; v[1] = x.y;
}

// Global stores, named as such: through a generic pointer the compiler must
// assume that each may change shared memory, and reads the column list, R - I and
// the next operands again after every one of them (a 4 x 16 tile took 6 us).
// Volatile: they stay before the barriers that publish them.
__device__ __forceinline__ void stg(float* p, float v) {
    asm volatile("st.global.f32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "f"(v));
}
__device__ __forceinline__ void stg(double* p, double v) {
    asm volatile("st.global.f64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "d"(v));
}

__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Rotation that annihilates s_pq: tan(theta) = b / (d + sgn(d) sqrt(d^2 + b^2)),
// d = s_qq - s_pp, b = 2 s_pq (the root of smaller magnitude of
// b t^2 + 2 d t - b = 0).  d and b are first scaled by a power of two so that
// the larger lies in [1, 2): no overflow, and b^2 underflows only where t = b / 2d
// to working accuracy.  Hardware reciprocal and reciprocal square root: the
// rotation only steers the pivot towards diagonal form, the accumulated R is
// re-orthonormalised before use, and the next sweep forms its Grams afresh.
__device__ __forceinline__ void rotation(float d, float apq, float& t, float& c, float& s) {
    const float b = 2.f * apq;
    const unsigned e = __float_as_uint(fmaxf(fabsf(d), fabsf(b))) & 0x7F800000u;
    const float sc = __uint_as_float(0x7F000000u - e);
    const float fd = d * sc, fb = b * sc;
    const float h = fmaf(fd, fd, fb * fb);
    t = fb * rcp_approx(fd + copysignf(h * rsqrt_approx(h), fd));
    c = rsqrt_approx(fmaf(t, t, 1.f));
    s = t * c;
}
// |s_pq| > eps sqrt(s_pp s_qq), roots of the hardware's accuracy, a root each: the
// product of two squared norms overflows from norms of 4e9 on (and then no pair
// was rotated: an SVT of a 90 x 100 matrix of norm 1e10 was off by 17 %)
__device__ __forceinline__ bool needs_rotation(float app, float aqq, float apq) {
    const float q = sqrt_approx(fabsf(app)) * sqrt_approx(fabsf(aqq));
    return fabsf(apq) > FLT_MIN && fabsf(apq) > FLT_EPSILON * q;
}
// non-negative norms ordered by their bits (a NaN sorts first: the order stays
// a permutation whatever the input holds)
__device__ __forceinline__ unsigned key_of(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ unsigned long long key_of(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}

// acc += (SR rows, column by column)^T (the same): lane (ti, tj) of 16 x 2
// holds the entries (ti + 16u, j0 + tj + 2v) of TI x TJ, so that 16-byte reads,
// each worth V rows of one column, meet no bank twice.
template <typename T, int TI, int TJ>
__device__ __forceinline__ void gram_rows(const T* st, int stride, int ti, int j0, T (&acc)[TI][TJ]) {
    constexpr int V = Cfg<T>::V;
    T part[TI][TJ];
#pragma unroll
    for (int u = 0; u < TI; ++u)
#pragma unroll
        for (int v = 0; v < TJ; ++v) part[u][v] = sizeof(T) == 4 ? T(0) : acc[u][v];
#pragma unroll
    for (int q = 0; q < Cfg<T>::SR; q += V) {
        T xi[TI][V];
#pragma unroll
        for (int u = 0; u < TI; ++u) lds16(st + (ti + 16 * u) * stride + q, xi[u]);
#pragma unroll
        for (int v = 0; v < TJ; ++v) {
            T xj[V];
            lds16(st + (j0 + 2 * v) * stride + q, xj);
#pragma unroll
            for (int e = 0; e < V; ++e)
#pragma unroll
                for (int u = 0; u < TI; ++u) part[u][v] = fma(xi[u][e], xj[e], part[u][v]);
        }
    }
#pragma unroll
    for (int u = 0; u < TI; ++u)
#pragma unroll
        for (int v = 0; v < TJ; ++v) acc[u][v] = sizeof(T) == 4 ? acc[u][v] + part[u][v] : part[u][v];
}
template <typename T, int TI, int TJ>
__device__ __forceinline__ void put_partial(T* part, int ti, int j0, const T (&acc)[TI][TJ]) {
#pragma unroll
    for (int u = 0; u < TI; ++u)
#pragma unroll
        for (int v = 0; v < TJ; ++v) part[(ti + 16 * u) * Smem<T>::PS + j0 + 2 * v] = acc[u][v];
}

// 256 threads: the partial Grams from chunks staged by the whole CTA, the next
// chunk's loads in flight during the products; two warps to a slot, half of
// the columns each (float64: two slots to a warp).  (Warps that stage their own rows and columns need no
// barrier, but three times the shared memory and more registers.)
template <typename T>
__device__ __forceinline__ void gram_staged(const Smem<T>& sm, T* stage) {
    constexpr int B2 = Smem<T>::B2, ST = Smem<T>::ST, TI = B2 / 16, PER = B2 * CHR / NT_MANY;
    constexpr int WPS = sizeof(T) == 4 ? 2 : 1, SPW = sizeof(T) == 4 ? 1 : 2, TJ = B2 / 2 / WPS;   // warps per slot, slots per warp
    const OsjDesc<T>& d = sm.d;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int slot = WPS == 2 ? warp & 3 : warp, j0 = (WPS == 2 ? (warp >> 2) * (B2 / 2) : 0) + (lane >> 4), ti = lane & 15;
    T* const buf = stage + Smem<T>::PART;
    const int frow = t % CHR, fcol = t / CHR;
    T pre[PER];
    auto fetch = [&](int ch) {
        const int row = ch * CHR + frow;
        const bool ok = row < d.L;
        const T* const base = d.X + row;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int gc = sm.cid[fcol + u * (NT_MANY / CHR)];
            pre[u] = (ok && gc >= 0) ? __ldcg(base + (int64_t)gc * d.ldx) : T(0);
        }
    };
    T acc[SPW][TI][TJ];
#pragma unroll
    for (int w = 0; w < SPW; ++w)
#pragma unroll
        for (int u = 0; u < TI; ++u)
#pragma unroll
            for (int v = 0; v < TJ; ++v) acc[w][u][v] = T(0);
    const int nch = (d.L + CHR - 1) / CHR;
    fetch(0);
    for (int ch = 0; ch < nch; ++ch) {
        T* const st = buf + (ch & 1) * (B2 * ST);
#pragma unroll
        for (int u = 0; u < PER; ++u) st[(fcol + u * (NT_MANY / CHR)) * ST + frow] = pre[u];
        __syncthreads();      // (the buffer's last readers passed the previous chunk's barrier)
        if (ch + 1 < nch) fetch(ch + 1);
#pragma unroll
        for (int w = 0; w < SPW; ++w) gram_rows<T, TI, TJ>(st + (slot + 8 * w) * Cfg<T>::SR, ST, ti, j0, acc[w]);
    }
#pragma unroll
    for (int w = 0; w < SPW; ++w) put_partial<T, TI, TJ>(stage + (slot + 8 * w) * B2 * Smem<T>::PS, ti, j0, acc[w]);
}

// what a pivot needs to know of its block (in registers)
template <typename T>
struct PivotCtx {
    T *X, *W;
    int ldx, ldw, L, p;
    T scale, tau, floor2, inv_scale;
    float ftau, ffloor;             // tau and floor2 relative to the scale
    T *stage, *panel, *wpanel;      // stage; kept columns of X and of W (512 threads)
    T* gpart;                       // clusterless: the team's partial Grams, else nullptr
    unsigned *team, *gave_up;       // and its arrivals
    int rank, split, member, stride, wstride;
    bool first_round;     // first round of the sweep: pairs inside the column blocks too
};

// 512 threads: the member's rows of the pivot columns into shared memory, all
// loads in flight together (an L2 load takes about 0.65 us); rows past L are zero.
// Local row (c own + j) SR + i is row 64 c + SR (member own + j) + i.
template <typename T>
__device__ __forceinline__ int global_row(int lr, int own, int member) {
    constexpr int SR = Cfg<T>::SR;
    const int g = lr / SR;
    return g / own * CHR + (member * own + g % own) * SR + lr % SR;
}
template <typename T>
__device__ __forceinline__ void load_panel(const PivotCtx<T>& d, const Smem<T>& sm, int own, int member) {
    constexpr int B2 = Smem<T>::B2, KB = B2 / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nr = (d.stride - Cfg<T>::V) / 32;            // 32-row groups
    for (int w = warp; w < nr * 2; w += NT_FEW / 32) {
        const int lr = (w >> 1) * 32 + lane, k0 = (w & 1) * KB;
        const int row = global_row<T>(lr, own, member);
        const bool ok = row < d.L;
        const T* const base = d.X + row;
        T* const dst = d.panel + lr;
        T pre[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            const int gc = sm.cid[k0 + k];
            pre[k] = (ok && gc >= 0) ? __ldcg(base + (int64_t)gc * d.ldx) : T(0);
        }
#pragma unroll
        for (int k = 0; k < KB; ++k) dst[(k0 + k) * d.stride] = pre[k];
    }
}

// 512 threads: the partial Grams of the member's slots from the kept columns into
// `part`, WPS warps to a slot with their shares of the columns (a split pivot's
// member has fewer slots and leaves the other warps out).
template <typename T, int WPS>
__device__ __forceinline__ void gram_slots(const PivotCtx<T>& d, int own, T* part) {
    constexpr int B2 = Smem<T>::B2, TI = B2 / 16, TJ = B2 / 2 / WPS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j = warp / WPS, j0 = (warp % WPS) * (B2 / WPS) + (lane >> 4), ti = lane & 15;
    if (j >= own) return;
    T acc[TI][TJ];
#pragma unroll
    for (int u = 0; u < TI; ++u)
#pragma unroll
        for (int v = 0; v < TJ; ++v) acc[u][v] = T(0);
    const int nch = (d.L + CHR - 1) / CHR;
#pragma unroll 1
    for (int c = 0; c < nch; ++c) gram_rows<T, TI, TJ>(d.panel + (c * own + j) * Cfg<T>::SR, d.stride, ti, j0, acc);
    put_partial<T, TI, TJ>(part + j * B2 * Smem<T>::PS, ti, j0, acc);
}
template <typename T>
__device__ __forceinline__ void gram_kept(const PivotCtx<T>& d, int own, T* part) {
    if constexpr (sizeof(T) == 4) {
        gram_slots<T, 4>(d, own, part);       // (more warps to a slot only read the same columns more often)
    } else {
        if (own == 16) gram_slots<T, 1>(d, own, part);
        else if (own == 8) gram_slots<T, 2>(d, own, part);
        else if (own == 4) gram_slots<T, 4>(d, own, part);
        else gram_slots<T, 8>(d, own, part);
    }
}

// Clusterless form: the CTAs of a block meet through its workspace, of
// unsigned integers first (arrivals of the block, CTAs that have left, given up,
// unused, arrivals of each team), then the partial Grams of every team, twice
// (a member may be one pivot ahead of the slowest reader).  The launch is
// cooperative, so the CTAs are all resident; a wait still gives up after some
// seconds, and with it every other.
constexpr int GRID_HEAD = 4;
constexpr int POLLS = 1 << 22;
__host__ __device__ constexpr size_t grid_head_words(int npairs) { return ((size_t)GRID_HEAD + npairs + 31) / 32 * 32; }

__device__ __forceinline__ unsigned poll(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(__cvta_generic_to_global(p)) : "memory");
    return v;
}
// all threads of the n CTAs that share `count` (zero before the first meeting)
__device__ __forceinline__ void meet(unsigned* count, unsigned n, unsigned* gave_up, int& fail) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned before = atomicAdd(count, 1u), target = before - before % n + n;
        int polls = 0;
        while ((int)(poll(count) - target) < 0) {
            if (++polls < POLLS && (polls % 64 != 0 || poll(gave_up) == 0)) continue;
            atomicExch(gave_up, 1u);
            fail = 1;
            break;
        }
        __threadfence();
    }
    __syncthreads();
}

// One row of 2b pivot columns times (R - I): x_j <- x_j + sum_k x_k (R - I)_kj,
// rows of R - I read by broadcast.  float32 uses the paired FMA (half the issue
// slots of the scalar one, which the broadcast reads then fill).
__device__ __forceinline__ void row_update(const float* R4, const float (&x)[32], int h, float (&o)[16]) {
    unsigned long long a[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) a[v] = 0ull;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        unsigned long long xx;
        asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x[k]));
        const ulonglong2* const r = reinterpret_cast<const ulonglong2*>(R4 + k * 32 + h * 16);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const ulonglong2 q = r[v];
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a[2 * v]) : "l"(xx), "l"(q.x));
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a[2 * v + 1]) : "l"(xx), "l"(q.y));
        }
    }
#pragma unroll
    for (int v = 0; v < 8; ++v) asm("mov.b64 {%0, %1}, %2;" : "=f"(o[2 * v]), "=f"(o[2 * v + 1]) : "l"(a[v]));
}
__device__ __forceinline__ void row_update(const double* R4, const double (&x)[16], int h, double (&o)[8]) {
#pragma unroll
    for (int v = 0; v < 8; ++v) o[v] = 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            double q[2];
            lds16(R4 + k * 16 + h * 8 + 2 * v, q);
            o[2 * v] = fma(x[k], q[0], o[2 * v]);
            o[2 * v + 1] = fma(x[k], q[1], o[2 * v + 1]);
        }
    }
}

// 512 threads: rows [row0, row0 + 32 RT) of kept columns times (R - I), columns
// h OW .. h OW + OW - 1, by one warp; a lane has rows row0 + lane + 32 i.  Every
// value of R - I is read (by broadcast) once for RT rows: with one row per lane
// the broadcast reads, two shared-memory cycles each, took twice the time of the
// FMAs they fed (5.4 us for 512 rows of a 32-column pivot).  store(i, v, value) receives row i's
// output column h OW + v.
template <int RT, typename Store>
__device__ __forceinline__ void tile_update(const float* R4, const float* cols, int stride, int h, Store store) {
    unsigned long long a[RT][8];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int v = 0; v < 8; ++v) a[i][v] = 0ull;
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
        ulonglong2 q[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) q[v] = reinterpret_cast<const ulonglong2*>(R4 + k * 32 + h * 16)[v];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            unsigned long long xx;
            asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(cols[k * stride + 32 * i]));
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a[i][2 * v]) : "l"(xx), "l"(q[v].x));
                asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a[i][2 * v + 1]) : "l"(xx), "l"(q[v].y));
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 8; ++v)
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            float o0, o1;
            asm("mov.b64 {%0, %1}, %2;" : "=f"(o0), "=f"(o1) : "l"(a[i][v]));
            store(i, 2 * v, cols[(h * 16 + 2 * v) * stride + 32 * i] + o0);
            store(i, 2 * v + 1, cols[(h * 16 + 2 * v + 1) * stride + 32 * i] + o1);
        }
}
template <int RT, typename Store>
__device__ __forceinline__ void tile_update(const double* R4, const double* cols, int stride, int h, Store store) {
    double a[RT][8];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int v = 0; v < 8; ++v) a[i][v] = 0.0;
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
        double q[8];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            double w[2];
            lds16(R4 + k * 16 + h * 8 + 2 * v, w);
            q[2 * v] = w[0];
            q[2 * v + 1] = w[1];
        }
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const double x = cols[k * stride + 32 * i];
#pragma unroll
            for (int v = 0; v < 8; ++v) a[i][v] = fma(x, q[v], a[i][v]);
        }
    }
#pragma unroll
    for (int v = 0; v < 8; ++v)
#pragma unroll
        for (int i = 0; i < RT; ++i) store(i, v, cols[(h * 8 + v) * stride + 32 * i] + a[i][v]);
}

// The inner rotations of a float64 pivot (sorted schedule), in float32 apart
// from the diagonal, which is kept as pairs of float32 so that the gaps of close
// columns are known to 2^-48.  A float64 operation takes 65 cycles and one warp
// instruction every 19 keeps the whole SM's unit busy: 32 us a pivot in float64,
// of 80.  The rotations only steer: what float32 leaves behind is 1e-7 of what
// was rotated away, found again by the next sweep's float64 Gram, while R is
// made orthogonal to float64 rounding before it is applied.  Up to two passes; the
// second is left out when no tangent was above 1e-6 (its square is below
// float32's own error by then).
__device__ __forceinline__ void inner_f64(Smem<double>& sm, double scale, double floor2, bool first_round) {
    constexpr int OB = Cfg<double>::OB, B2 = 2 * OB, LS = Cfg<double>::LS;
    const int t = threadIdx.x;
    float* const S2 = reinterpret_cast<float*>(sm.S[1]);       // two buffers
    float* const R = reinterpret_cast<float*>(sm.G);
    float* const lo2 = R + B2 * LS;                            // low parts of the diagonal, two buffers
    static_assert(B2 * LS + 2 * B2 <= 2 * B2 * B2, "R and the low parts in the place of R^T R");
    // the largest column's square to 2^60: entries down to 1e-56 of it are normal
    const int e = 1023 + 60 - ((__double2hiint(scale) >> 20) - 1023);
    const int ec = min(max(e, 1), 2045);
    const double sc = __hiloint2double(ec << 20, 0), inv_sc = __hiloint2double((2046 - ec) << 20, 0);
    if (t < B2 * B2) {
        const int i = t / B2, j = t % B2;
        const double v = sm.S[0][i * LS + j] * sc;
        const float f = (float)v;
        S2[i * LS + j] = f;
        R[i * LS + j] = i == j ? 1.f : 0.f;
        if (i == j) lo2[i] = (float)(v - (double)f);
    }
    const float ffloor = (float)(floor2 * sc);
    __syncthreads();
    if (t < OB * OB) {
        const int k = t % OB, l = t / OB;
        int cur = 0, rotated = 0;
        const int r_first = first_round ? -(OB - 1) : 0;
        for (int pass = 0; pass < 2; ++pass) {
            int big = 0;
            for (int r = r_first; r < OB; ++r) {
                int pk, qk, pl, ql;
                if (r >= 0) {
                    pk = k; qk = OB + ((k + r) & (OB - 1));
                    pl = l; ql = OB + ((l + r) & (OB - 1));
                } else {
                    // pairs inside column block a (first half) and c
                    constexpr int H = OB / 2;
                    const int rr = r + OB - 1, ok = k < H ? 0 : OB, ol = l < H ? 0 : OB;
                    pk = ok + circle_item(k & (H - 1), rr, OB); qk = ok + circle_item(OB - 1 - (k & (H - 1)), rr, OB);
                    pl = ol + circle_item(l & (H - 1), rr, OB); ql = ol + circle_item(OB - 1 - (l & (H - 1)), rr, OB);
                }
                const float* const S = S2 + cur * B2 * LS;
                float* const D = S2 + (cur ^ 1) * B2 * LS;
                const float* const lo = lo2 + cur * B2;
                float* const lo_new = lo2 + (cur ^ 1) * B2;
                const float app = S[pk * LS + pk], aqq = S[qk * LS + qk], apq = S[pk * LS + qk];
                const float lp = lo[pk], lq = lo[qk];
                const float s_pu = S[pk * LS + pl], s_pv = S[pk * LS + ql], s_qu = S[qk * LS + pl], s_qv = S[qk * LS + ql];
                const float x0 = R[k * LS + pl], y0 = R[k * LS + ql];
                const float x1 = R[(k + OB) * LS + pl], y1 = R[(k + OB) * LS + ql];
                float tk, ck, sk;
                rotation((aqq - app) + (lq - lp), apq, tk, ck, sk);
                const bool act = fabsf(apq) > FLT_MIN &&
                                 fabsf(apq) > (float)DBL_EPSILON * (sqrt_approx(fabsf(app)) * sqrt_approx(fabsf(aqq)));
                tk = act ? tk : 0.f;
                ck = act ? ck : 1.f;
                sk = act ? sk : 0.f;
                rotated |= act;
                big |= act && fabsf(apq) > ffloor && fabsf(tk) > 1e-6f;
                const float clr = __shfl_sync(0xffffffffu, ck, l), slr = __shfl_sync(0xffffffffu, sk, l);
                const float r_pu = fmaf(ck, s_pu, -(sk * s_qu)), r_pv = fmaf(ck, s_pv, -(sk * s_qv));
                const float r_qu = fmaf(sk, s_pu, ck * s_qu), r_qv = fmaf(sk, s_pv, ck * s_qv);
                float d_pu = fmaf(clr, r_pu, -(slr * r_pv)), d_pv = fmaf(slr, r_pu, clr * r_pv);
                float d_qu = fmaf(clr, r_qu, -(slr * r_qv)), d_qv = fmaf(slr, r_qu, clr * r_qv);
                if (k == l) {
                    // the pair's own block: diagonal +- t s_pq in pairs of float32
                    const float x = tk * apq;
                    const float hp = app - x, bp = hp - app, ep = ((app - (hp - bp)) + (-x - bp)) + lp;
                    const float hq = aqq + x, bq = hq - aqq, eq = ((aqq - (hq - bq)) + (x - bq)) + lq;
                    d_pu = hp + ep; lo_new[pk] = ep - (d_pu - hp);
                    d_qv = hq + eq; lo_new[qk] = eq - (d_qv - hq);
                    d_pv = act ? 0.f : s_pv;
                    d_qu = act ? 0.f : s_qu;
                }
                D[pk * LS + pl] = d_pu;
                D[pk * LS + ql] = d_pv;
                D[qk * LS + pl] = d_qu;
                D[qk * LS + ql] = d_qv;
                R[k * LS + pl] = fmaf(clr, x0, -(slr * y0));
                R[k * LS + ql] = fmaf(slr, x0, clr * y0);
                R[(k + OB) * LS + pl] = fmaf(clr, x1, -(slr * y1));
                R[(k + OB) * LS + ql] = fmaf(slr, x1, clr * y1);
                cur ^= 1;
                if (r == OB - 1) {
                    if (big) sm.sig[pass] = 1;
                    if (rotated) sm.rot = 1;
                }
                asm volatile("bar.sync 1, %0;" ::"n"(OB * OB) : "memory");
            }
            if (!sm.sig[pass]) break;
        }
        if (t == 0) sm.cur = cur;
    }
    __syncthreads();
    if (t < B2 * B2) {
        const int i = t / B2, j = t % B2;
        sm.R[i * LS + j] = (double)R[i * LS + j];
        if (i == j) sm.S[0][i * LS + i] = ((double)S2[sm.cur * B2 * LS + i * LS + i] + (double)lo2[sm.cur * B2 + i]) * inv_sc;
    }
}

// One pivot (logical column blocks a and c) of one round: Gram, measure,
// rotation.  Returns the convergence measure of the pivot (CTA-uniform);
// top_a / top_c receive the two largest squared norms of the column blocks.
template <typename T, int NT, bool KEEP>
__device__ T osj_pivot(Smem<T>& sm, cg::cluster_group& cl, const PivotCtx<T>& cx, int a, int c, T* top_a, T* top_c) {
    constexpr int OB = Cfg<T>::OB, B2 = 2 * OB, LS = Cfg<T>::LS, NW = NT / 32;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int split = NT == NT_MANY ? 1 : cx.split, member = NT == NT_MANY ? 0 : cx.member;

    if (t < B2) {
        const int pos = t < OB ? a * OB + t : c * OB + (t - OB);
        sm.cid[t] = pos < sm.d.p ? (KEEP ? pos : __ldcg(sm.d.ord + pos)) : -1;
    }
    if (t == 32) { sm.sig[0] = 0; sm.sig[1] = 0; sm.rot = 0; }
    __syncthreads();

    // ---- 1. Gram
    constexpr int NSLOT = Cfg<T>::NSLOT;
    const int own = NSLOT / split;
    if constexpr (NT == NT_MANY) {
        gram_staged<T>(sm, reinterpret_cast<T*>(&sm + 1));
        __syncthreads();
    } else {
        load_panel<T>(cx, sm, own, member);
        __syncthreads();
        const bool shared = split == 1 || !cx.gpart;
        gram_kept<T>(cx, own, shared ? cx.stage : cx.gpart + member * own * B2 * Smem<T>::PS);
        if (split == 1) __syncthreads();
        else if (shared) cl.sync();
        else meet(cx.team, (unsigned)split, cx.gave_up, sm.fail);
    }
    for (int e = t; e < B2 * B2; e += NT) {
        const int i = e / B2, j = e % B2;
        T p[NSLOT];
        constexpr int SLOT = B2 * Smem<T>::PS;
        const int at = i * Smem<T>::PS + j;
        const T* const mem = cx.gpart + at;
        const T* const here = reinterpret_cast<T*>(&sm + 1) + at;
        if (NT == NT_FEW && split > 1 && cx.gpart) {
#pragma unroll
            for (int sl = 0; sl < NSLOT; ++sl) p[sl] = __ldcg(mem + sl * SLOT);
        } else if (NT == NT_FEW && split > 1) {
#pragma unroll
            for (int sl = 0; sl < NSLOT; ++sl)
                p[sl] = *cl.map_shared_rank(here + (sl % own) * SLOT, cx.rank - member + sl / own);
        } else {
#pragma unroll
            for (int sl = 0; sl < NSLOT; ++sl) p[sl] = here[sl * SLOT];
        }
        T sum = p[0];
#pragma unroll
        for (int sl = 1; sl < NSLOT; ++sl) sum += p[sl];
        sm.S[0][i * LS + j] = sum;
        sm.R[i * LS + j] = (i == j) ? T(1) : T(0);
    }
    __syncthreads();

    // ---- 2. convergence measure before rotating: how much the rotation this
    //      pair still needs could change J = U max(Sigma - tau, 0) V^T,
    //      relative to the largest singular value.  For columns of norms a, b
    //      an unresolved rotation of tangent t moves J by about t |f(a) - f(b)|
    //      (f(s) = max(s - tau, 0) is 1-Lipschitz, so |a - b| bounds it), plus
    //      tau theta when both lie above tau (the pair then enters J as
    //      A - tau U V^T and theta = |s_ij| / (a b) is its angle defect).
    //      A pair with a^2 + b^2 <= tau^2 has its own two singular values below
    //      tau, but many such columns together may not: a set of them stays
    //      below tau, whatever its rotation, while every max(a^2, b^2) + p |s_ij|
    //      <= tau^2 (Gershgorin's bound on its Gram), which is what the sorted
    //      schedule asks of them; the kept schedule leaves them out (they are
    //      rotated with the larger columns of their pivots).
    //      Columns below the rounding floor (~4 eps of the largest) are noise
    //      and skipped.  A `strict` matrix (the block whose kept left singular
    //      subspace the C step projects onto) also needs that subspace itself:
    //      pairs that straddle tau are measured by t alone.
    const T tau = cx.tau, tau2 = tau * tau;
    using M = std::conditional_t<KEEP, T, float>;
    M offm = M(0);
    if constexpr (KEEP) {
        const T smax = sqrt(cx.scale);
        const T inv_smax = T(1) / (smax + num<T>::tiny());
        for (int e = t; e < B2 * B2; e += NT) {
            const int i = e % B2, j = e / B2;
            const T sii = sm.S[0][i * LS + i], sjj = sm.S[0][j * LS + j];
            if (i < j && sii > cx.floor2 && sjj > cx.floor2 && sii + sjj > tau2) {
                const T sij = fabs(sm.S[0][i * LS + j]);
                const T na = sqrt(sii), nb = sqrt(sjj);
                const T hd = T(0.5) * fabs(sii - sjj);
                const T tn = sij / (hd + sqrt(hd * hd + sij * sij) + num<T>::tiny());
                T mm;
                if (na > tau && nb > tau) mm = tn * fabs(na - nb) + tau * sij / (na * nb);
                else if (na > tau || nb > tau)
                    mm = sm.d.strict ? tn * (cx.scale > 0 ? smax : T(1)) : tn * fabs(na - nb);
                else mm = tn * (sqrt(sii + sjj) - tau);
                offm = fmax(offm, mm * inv_smax);
            }
        }
    } else {
        // the differences are taken in T, the rest in float32 on values relative
        // to the largest column: the measure only steers the sweeps
        const T inv_scale = cx.inv_scale;
        const float ftau = cx.ftau;
        for (int e = t; e < B2 * B2; e += NT) {
            const int j = e % B2, i = e / B2;
            if (i >= j) continue;
            const T sii = sm.S[0][i * LS + i], sjj = sm.S[0][j * LS + j];
            const float a2 = (float)(sii * inv_scale), b2 = (float)(sjj * inv_scale);
            if (a2 > cx.ffloor && b2 > cx.ffloor) {
                const T sij = fabs(sm.S[0][i * LS + j]);
                const float fs = (float)(sij * inv_scale), df = fabsf((float)((sii - sjj) * inv_scale));
                const float na = sqrtf(a2), nb = sqrtf(b2), gap = df / (na + nb);       // |na - nb|
                // tangent 2 s / (|a^2 - b^2| + sqrt((a^2 - b^2)^2 + 4 s^2)), scaled against underflow
                const float m = fmaxf(df, 2.f * fs), mi = m > 0.f ? 1.f / m : 0.f;
                const float u = df * mi, w = 2.f * fs * mi;
                const float tn = w / (u + sqrtf(fmaf(u, u, w * w)) + FLT_MIN);
                float mm;
                if (sii + sjj <= tau2) {
                    const T g = fmax(sii, sjj) + T(sm.d.p) * sij;
                    const float fg = (float)((g - tau2) * inv_scale);
                    mm = fg / (sqrtf((float)(g * inv_scale)) + ftau);
                } else if (sii > tau2 && sjj > tau2) mm = tn * gap + ftau * fs / (na * nb);
                else if (sii > tau2 || sjj > tau2) mm = sm.d.strict ? tn : tn * gap;
                else mm = tn * (float)((sii + sjj - tau2) * inv_scale) / (sqrtf(a2 + b2) + ftau);
                offm = fmaxf(offm, mm);
            }
        }
    }
    offm = warp_max(offm);
    M* const red = reinterpret_cast<M*>(sm.red);
    if (lane == 0) red[warp] = offm;
    __syncthreads();
    M mxm = M(0);
#pragma unroll
    for (int w = 0; w < NW; ++w) mxm = fmax(mxm, red[w]);
    const T mx = (T)mxm;

    // two largest diagonal entries of each column block (read by the next
    // rounds' skip test; member 0 writes them)
    const T* Sd = sm.S[0];
    auto tops = [&]() {
        if (member == 0 && (t == 0 || t == 32)) {
            T n1 = T(0), n2 = T(0);
            const int o = t == 0 ? 0 : OB;
            for (int i = 0; i < OB; ++i) {
                const T v = Sd[(o + i) * LS + o + i];
                if (!(v <= n1)) { n2 = n1; n1 = v; }      // a NaN counts as large
                else if (!(v <= n2)) n2 = v;
            }
            T* const dst = t == 0 ? top_a : top_c;
            dst[0] = n1;
            dst[1] = n2;
        }
    };
    // a pivot already orthogonal to a few eps needs no rotation (4 eps in
    // float32: on data with one dominant singular value the measure, relative
    // to the largest column, must resolve pairs well below it)
    if (mx <= (sizeof(T) == 4 ? T(4) : T(16)) * num<T>::eps()) {
        tops();
        __syncthreads();      // cid and S are rewritten by the next pivot
        return mx;
    }

    // 512 threads: the first rows of W are copied to shared memory while the pivot
    // rotates (split members take alternate 32-row groups), as 16-byte asynchronous
    // copies: through registers, 32 a thread, the copy and its spills took 2.3 us.
    // (Rows past p of the last group are read, W being padded, and not used.)
    const int wchunks = ((cx.p + 31) / 32 - member + split - 1) / split, wrows = wchunks * 32;
    auto wrow = [&](int lw) { return ((lw / 32) * split + member) * 32 + lw % 32; };
    auto fetch_w = [&](int w0) {
        if constexpr (NT == NT_FEW) {
            constexpr int V = Cfg<T>::V, PER = 32 / V;
            static_assert(PER * B2 == 256, "256 copies to a group of 32 rows");
            const int wg = min(wchunks - w0 / 32, WROWS / 32), k = (t & 255) / PER, v = (t & 255) % PER * V;
            const int gc = sm.cid[k];
            const T* const src = cx.W + (int64_t)max(gc, 0) * cx.ldw + v;
            const unsigned dst = (unsigned)__cvta_generic_to_shared(cx.wpanel + k * cx.wstride + v);
            for (int g = t >> 8; g < wg; g += NT / 256)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + g * 32 * (unsigned)sizeof(T)),
                             "l"(__cvta_generic_to_global(src + wrow(w0 + g * 32))), "r"(gc >= 0 ? 16 : 0) : "memory");
        }
    };
    fetch_w(0);

    // ---- 3. rotate the pivot Gram towards diagonal form.  Thread (k, l) of
    //      b x b owns the 2 x 2 sub-block of pairs k and l: it reads the old S,
    //      works out pair k's rotation itself, takes pair l's from the lane that
    //      has it, and writes the other S buffer, so a round costs one barrier
    //      of these b^2 threads and one chain of shared read, rotation, write
    //      (0.25 us; 0.7 us with a barrier on either side of the rotations).
    //      Sorted: 62 rounds in the first round of a sweep, else 32, or half of
    //      that when the first pass found only small angles (no tangent above
    //      3e-4: what the second would still find is the square of that).  Kept: 31 rounds.
    if constexpr (sizeof(T) == 8) {
        inner_f64(sm, cx.scale, cx.floor2, cx.first_round);
    } else if (t < OB * OB) {
        const int k = t % OB, l = t / OB;
        int cur = 0, rotated = 0;
        int pk = k, qk = B2 - 1 - k, pl = l, ql = B2 - 1 - l;       // the circle method's round 0
        const int r_first = KEEP ? 0 : cx.first_round ? -(OB - 1) : 0, r_end = KEEP ? B2 - 1 : OB;
        for (int pass = 0; pass < (KEEP ? 1 : 2); ++pass) {
            int big = 0;
            for (int r = r_first; r < r_end; ++r) {
                if (KEEP) {
                    // (moved on at the end of the round)
                } else if (r >= 0) {
                    pk = k; qk = OB + ((k + r) & (OB - 1));
                    pl = l; ql = OB + ((l + r) & (OB - 1));
                } else {
                    // pairs inside column block a (first half) and c
                    constexpr int H = OB / 2;
                    const int rr = r + OB - 1, ok = k < H ? 0 : OB, ol = l < H ? 0 : OB;
                    pk = ok + circle_item(k & (H - 1), rr, OB); qk = ok + circle_item(OB - 1 - (k & (H - 1)), rr, OB);
                    pl = ol + circle_item(l & (H - 1), rr, OB); ql = ol + circle_item(OB - 1 - (l & (H - 1)), rr, OB);
                }
                const T* const S = sm.S[cur];
                T* const D = sm.S[cur ^ 1];
                const T app = S[pk * LS + pk], aqq = S[qk * LS + qk], apq = S[pk * LS + qk];
                const T s_pu = S[pk * LS + pl], s_pv = S[pk * LS + ql], s_qu = S[qk * LS + pl], s_qv = S[qk * LS + ql];
                const T x0 = sm.R[k * LS + pl], y0 = sm.R[k * LS + ql];
                const T x1 = sm.R[(k + OB) * LS + pl], y1 = sm.R[(k + OB) * LS + ql];
                // (always computed, then selected: a branch costs more than the
                // few lanes it would spare)
                T ck, sk;
                bool act;
                if constexpr (KEEP) {
                    act = fabs(apq) > num<T>::tiny() && above_eps_root(fabs(apq), fabs(app * aqq));
                    jacobi_rotation<T>(app, aqq, apq, ck, sk);
                } else {
                    act = needs_rotation(app, aqq, apq);
                    float tn;
                    rotation(aqq - app, apq, tn, ck, sk);
                }
                ck = act ? ck : T(1);
                sk = act ? sk : T(0);
                rotated |= act;
                if (!KEEP) big |= act && fabs(apq) > cx.floor2 && fabs(sk) > T(3e-4) * ck;
                const T clr = __shfl_sync(0xffffffffu, ck, l), slr = __shfl_sync(0xffffffffu, sk, l);
                // (fused multiply-adds written out: which product of a sum of two is
                // rounded first is part of the kept schedule's arithmetic)
                const T r_pu = fma(ck, s_pu, -(sk * s_qu)), r_pv = fma(ck, s_pv, -(sk * s_qv));
                const T r_qu = fma(sk, s_pu, ck * s_qu), r_qv = fma(sk, s_pv, ck * s_qv);
                // the rotated pair's own off-diagonal entries are zero by
                // construction (to the rounding of the next fresh Gram)
                const bool zero = k == l && sk != T(0);
                D[pk * LS + pl] = fma(clr, r_pu, -(slr * r_pv));
                D[pk * LS + ql] = zero ? T(0) : fma(slr, r_pu, clr * r_pv);
                D[qk * LS + pl] = zero ? T(0) : fma(clr, r_qu, -(slr * r_qv));
                D[qk * LS + ql] = fma(slr, r_qu, clr * r_qv);
                sm.R[k * LS + pl] = fma(clr, x0, -(slr * y0));
                sm.R[k * LS + ql] = fma(slr, x0, clr * y0);
                sm.R[(k + OB) * LS + pl] = fma(clr, x1, -(slr * y1));
                sm.R[(k + OB) * LS + ql] = fma(slr, x1, clr * y1);
                cur ^= 1;
                if (KEEP) {
                    pk = k ? (pk == B2 - 1 ? 1 : pk + 1) : 0;
                    pl = l ? (pl == B2 - 1 ? 1 : pl + 1) : 0;
                    qk = qk == B2 - 1 ? 1 : qk + 1;
                    ql = ql == B2 - 1 ? 1 : ql + 1;
                }
                if (r == r_end - 1) {
                    if (big) sm.sig[pass] = 1;
                    if (rotated) sm.rot = 1;
                }
                asm volatile("bar.sync 1, %0;" ::"n"(OB * OB) : "memory");
            }
            if (!KEEP && !sm.sig[pass]) break;
        }
        if (t == 0) sm.cur = cur;
    }
    __syncthreads();
    if (sizeof(T) == 4) Sd = sm.S[sm.cur];
    tops();
    if (!sm.rot) {
        asm volatile("cp.async.wait_all;" ::: "memory");      // (W's place is the next pivot's stage)
        __syncthreads();
        return mx;
    }

    // R is a product of some hundred plane rotations, orthogonal only to
    // ~sqrt(count) eps; one Newton-Schulz step R <- R (3I - R^T R)/2 restores
    // orthogonality to ~eps^2 before R touches X and W (applied to graded
    // columns the defect would mix eps-sized parts of the large columns into
    // the small ones).  Float64: R comes from float32 rotations, with E = I - R^T R
    // up to some 1e-6, and R (I - E)^(-1/2) is taken to second order, R + R (E / 2 +
    // 3/8 E^2), which leaves E^3; E^2 in float32 is good to 1e-19.
    // The rotation is applied in update form, x_j <- x_j + sum_k x_k (R - I)_kj:
    // once the sweeps have converged R - I is tiny and so is the rounding it
    // adds, instead of a fresh eps |x| at every application.
    constexpr int PE = B2 * B2 / 256;             // consecutive entries of a row per thread
    const int ni = t * PE / B2, nj = t * PE % B2;
    float* const Ef = reinterpret_cast<float*>(sm.S[1]);      // (float64; the rotations' S is done with)
    if (t < 256) {
        T g[PE];
#pragma unroll
        for (int u = 0; u < PE; ++u) g[u] = sizeof(T) == 8 && ni == nj + u ? T(-1) : T(0);
#pragma unroll 8
        for (int k = 0; k < B2; ++k) {
            const T x = sm.R[k * LS + ni];
#pragma unroll
            for (int u = 0; u < PE; ++u) g[u] = fma(x, sm.R[k * LS + nj + u], g[u]);
        }
#pragma unroll
        for (int u = 0; u < PE; ++u) {
            sm.G[ni * B2 + nj + u] = g[u];
            if (sizeof(T) == 8) Ef[ni * B2 + nj + u] = (float)g[u];
        }
    }
    __syncthreads();
    if constexpr (sizeof(T) == 8) {
        if (t < 256) {
            float e2 = 0.f;
#pragma unroll
            for (int k = 0; k < B2; ++k) e2 = fmaf(Ef[ni * B2 + k], Ef[k * B2 + nj], e2);
            sm.G[t] = fma(T(-0.5), sm.G[t], (T)(0.375f * e2));
        }
        __syncthreads();
    }
    if (t < 256) {
        T y[PE];
#pragma unroll
        for (int u = 0; u < PE; ++u) y[u] = T(0);
#pragma unroll 8
        for (int k = 0; k < B2; ++k) {
            const T x = sm.R[ni * LS + k];
#pragma unroll
            for (int u = 0; u < PE; ++u) y[u] = fma(x, sm.G[k * B2 + nj + u], y[u]);
        }
#pragma unroll
        for (int u = 0; u < PE; ++u) {
            const T rr = sm.R[ni * LS + nj + u], one = ni == nj + u ? T(1) : T(0);
            if (sizeof(T) == 8) {
                sm.R4[ni * B2 + nj + u] = (rr - one) + y[u];
            } else {
                const T rn = fma(T(1.5), rr, T(-0.5) * y[u]);
                sm.R4[ni * B2 + nj + u] = rn - one;
            }
        }
    }
    __syncthreads();

    // ---- 4. X_P <- X_P R and W_P <- W_P R
    constexpr int OW = 8 * (8 / sizeof(T));       // output columns at a time: 16 floats, 8 doubles
    static_assert(B2 == 2 * OW, "two halves");
    if constexpr (NT == NT_MANY) {
        // the rows of X, then those of W, in one sequence from L2, a row's 2b
        // pivot columns in a thread's registers
        const OsjDesc<T>& d = sm.d;
        const int rows = d.L + d.p;
        for (int r0 = 0; r0 < rows; r0 += NT) {
            const int row = r0 + t;
            const bool ok = row < rows, isx = row < d.L;
            if (r0 + warp * 32 >= rows) break;
            T* const base = isx ? d.X + row : d.W + (row - d.L);
            const int ld = isx ? d.ldx : d.ldw;
            T x[B2];
#pragma unroll
            for (int k = 0; k < B2; ++k) {
                const int gc = sm.cid[k];
                x[k] = (ok && gc >= 0) ? __ldcg(base + (int64_t)gc * ld) : T(0);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                T o[OW];
                row_update(sm.R4, x, h, o);
#pragma unroll
                for (int v = 0; v < OW; ++v) {
                    const int gc = sm.cid[h * OW + v];
                    if (ok && gc >= 0) base[(int64_t)gc * ld] = x[h * OW + v] + o[v];
                }
            }
        }
    } else {
        // from shared memory, one warp per tile of RT 32-row groups and half
        // the columns: the tiles of X first, then those of the W rows fetched above
        // (W rows past the first WROWS follow in turn)
        constexpr int RT = sizeof(T) == 4 ? 4 : 1;
        const int xg = (cx.stride - Cfg<T>::V) / 32, lrows = local_rows<T>(cx.L, split);
        for (int w0 = 0; w0 < wrows || w0 == 0; w0 += WROWS) {
            const int wg = min(wchunks - w0 / 32, WROWS / 32);
            if (w0 > 0) fetch_w(w0);
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            const int xt = w0 == 0 ? (xg + RT - 1) / RT : 0, wt = (wg + RT - 1) / RT;
            for (int tile = warp; tile < 2 * (xt + wt); tile += NT / 32) {
                const int h = tile & 1, g0 = tile / 2 < xt ? tile / 2 * RT : (tile / 2 - xt) * RT;
                int gcs[OW];
#pragma unroll
                for (int v = 0; v < OW; ++v) gcs[v] = sm.cid[h * OW + v];
                if (tile / 2 < xt) {
                    tile_update<RT>(sm.R4, cx.panel + g0 * 32 + lane, cx.stride, h, [&](int i, int v, T val) {
                        const int lr = (g0 + i) * 32 + lane, row = global_row<T>(lr, own, member);
                        if (lr < lrows && row < cx.L && gcs[v] >= 0) stg(cx.X + (int64_t)gcs[v] * cx.ldx + row, val);
                    });
                } else {
                    tile_update<RT>(sm.R4, cx.wpanel + g0 * 32 + lane, cx.wstride, h, [&](int i, int v, T val) {
                        const int row = wrow(w0 + (g0 + i) * 32 + lane);
                        if (g0 + i < wg && row < cx.p && gcs[v] >= 0) stg(cx.W + (int64_t)gcs[v] * cx.ldw + row, val);
                    });
                }
            }
            if (w0 + WROWS < wrows) __syncthreads();
        }
    }
    __syncthreads();
    return mx;
}

// One cluster per matrix (blockIdx.y).  `off` holds three slots per matrix
// (one per sweep, reused every third sweep).
// With `quad_exit`, a sweep whose measure o (taken before its rotations)
// satisfies 16 o^2 <= tol ends the loop without a confirming sweep: cyclic
// Jacobi converges quadratically near the end (the off-diagonal part after a
// sweep is O(o^2)), so the rotations of that sweep already bring the matrix
// below the tolerance.
template <typename T, int NT, bool KEEP>
__global__ void __launch_bounds__(NT, NT == NT_MANY ? 3 : 1) osj_svd(const OsjDesc<T>* __restrict__ descs, int sweeps, T tol,
                                              int* __restrict__ sweeps_run, int quad_exit, int split, int grid,
                                              const int* __restrict__ list) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem<T>& sm = *reinterpret_cast<Smem<T>*>(smem_raw);
    constexpr int OB = Cfg<T>::OB, NW = NT / 32;
    const int mat = list ? list[blockIdx.y] : (int)blockIdx.y;
    if (threadIdx.x == 0) sm.d = descs[mat];
    __syncthreads();
    const OsjDesc<T>& d = sm.d;
    if (d.active && *d.active == 0) return;     // uniform over the cluster
    cg::cluster_group cl = cg::this_cluster();
    const bool clusterless = NT == NT_FEW && grid;
    const int rank = (int)blockIdx.x, csize = (int)gridDim.x;      // (a cluster spans the grid's x)
    const int team = rank / split, nteams = csize / split;
    const int nb = 2 * ((d.p + 2 * OB - 1) / (2 * OB)), npairs = nb / 2;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    T* const nrm = d.cols;                      // squared column norms
    T* const top = d.cols + d.pp;               // 2 parities x nb x 2 largest norms
    if (rank == 0 && t == 0) { d.off[0] = T(0); d.off[1] = T(0); d.off[2] = T(0); }
    PivotCtx<T> cx;
    cx.X = d.X; cx.W = d.W;
    cx.ldx = (int)d.ldx; cx.ldw = (int)d.ldw; cx.L = d.L; cx.p = d.p;
    cx.rank = rank; cx.split = split; cx.member = rank % split;
    cx.stage = reinterpret_cast<T*>(&sm + 1);
    cx.stride = panel_stride<T>(d.L, split);
    cx.wstride = wpanel_stride<T>(d.p, split);
    if (NT == NT_FEW) {
        // partial Grams | W (over them unless split) | X
        constexpr int B2 = 2 * OB;
        cx.wpanel = split > 1 ? cx.stage + Smem<T>::PART : cx.stage;
        cx.panel = cx.stage + (split > 1 ? Smem<T>::PART + B2 * cx.wstride : max(Smem<T>::PART, B2 * cx.wstride));
    }
    // clusterless: the workspace
    unsigned* const head = static_cast<unsigned*>(d.grid);
    constexpr int GP = Cfg<T>::NSLOT * 2 * OB * Smem<T>::PS;        // a team's partial Grams
    T* const gparts = clusterless ? reinterpret_cast<T*>(head + grid_head_words(npairs)) + (size_t)team * 2 * GP : nullptr;
    cx.gpart = gparts;
    cx.gave_up = head + 2;
    cx.team = head + GRID_HEAD + team;
    if (t == 0) sm.fail = clusterless && poll(head + 2) != 0;
    __syncthreads();
    if (sm.fail) return;
    auto sync_block = [&]() {
        if (clusterless) meet(head, (unsigned)csize, head + 2, sm.fail);
        else cl.sync();
    };
    int flip = 0;
    cx.tau = d.mu ? (T)(1.0 / *d.mu) : T(0);
    // scaled off-diagonals below ~64 eps are at the rounding level of the
    // fresh pivot Grams
    const T t_eff = fmax(tol, T(64) * num<T>::eps());
    int par = 0;          // parity of the round: which copy of `top` it reads
    for (int sw = 0; sw < sweeps; ++sw) {
        if (KEEP ? sw == 0 : sw <= 4 && sw % 2 == 0) {
            // squared norms, a warp per column
            for (int j = rank * NW + warp; j < d.p; j += csize * NW) {
                const T* const x = d.X + j * d.ldx;
                T acc = T(0);
                for (int i = lane; i < d.L; i += 32) {
                    const T v = __ldcg(x + i);
                    acc = fma(v, v, acc);
                }
                acc = warp_sum(acc);
                if (lane == 0) nrm[j] = acc;
            }
            sync_block();
            // each column's place in the order: how many come before it
            constexpr int TS = 2 * OB * Smem<T>::PS;
            T* const stage = reinterpret_cast<T*>(&sm + 1);
            for (int jb = rank * NT; !KEEP && jb < d.p; jb += csize * NT) {
                const int j = jb + t;
                const auto kj = key_of(j < d.p ? __ldcg(nrm + j) : T(0));
                int before = 0;
                for (int i0 = 0; i0 < d.p; i0 += TS) {
                    const int cnt = min(TS, d.p - i0);
                    __syncthreads();
                    for (int i = t; i < cnt; i += NT) stage[i] = __ldcg(nrm + i0 + i);
                    __syncthreads();
                    for (int i = 0; i < cnt; ++i) {
                        const auto ki = key_of(stage[i]);
                        before += (ki > kj || (ki == kj && i0 + i < j)) ? 1 : 0;
                    }
                }
                if (j < d.p) d.ord[before] = j;
            }
            if (!KEEP) sync_block();
            if (clusterless && sm.fail) break;                 // (the order may be incomplete)
            // the two largest norms of every column block
            if (rank == 0)
                for (int b = t; b < nb; b += NT) {
                    T n1 = T(0), n2 = T(0);
                    for (int q = 0; q < OB; ++q) {
                        const int pos = b * OB + q;
                        if (pos >= d.p || (!KEEP && q >= 2)) break;
                        const T v = __ldcg(nrm + (KEEP ? pos : __ldcg(d.ord + pos)));
                        if (!(v <= n1)) { n2 = n1; n1 = v; }
                        else if (!(v <= n2)) n2 = v;
                    }
                    top[(par * nb + b) * 2] = n1;
                    top[(par * nb + b) * 2 + 1] = n2;
                }
            sync_block();
            if (sw == 0) {
                // the largest column: the scale of the measure and of the rounding floor
                T mx = T(0);
                for (int b = lane; b < nb; b += 32) mx = fmax(mx, __ldcg(top + 2 * b));
                cx.scale = warp_max(mx);
                const T noise = T(4) * num<T>::eps();
                cx.floor2 = noise * noise * cx.scale + num<T>::tiny();
                cx.inv_scale = T(1) / (cx.scale + num<T>::tiny());
                cx.ftau = (float)(cx.tau * sqrt(cx.inv_scale));
                cx.ffloor = (float)(cx.floor2 * cx.inv_scale);
            }
        }
        T mine = T(0);
        for (int r = 0; r < nb - 1; ++r) {
            cx.first_round = r == 0;
            const T* const ti = top + par * nb * 2;
            T* const to = top + (par ^ 1) * nb * 2;
            // Every warp lists the pivots that need work, 32 pairs at a time,
            // and the teams take them in turn.  A pair of column blocks is
            // skipped when no two of its columns reach a^2 + b^2 > tau^2 or when
            // at most one of them is above the rounding floor: its measure
            // would be zero.  The norms are one rotation old at most and good
            // to a few eps of the column block's largest, hence the margins.
            // (Sorted: nor does any pair come near Gershgorin's bound.  Its root is
            // taken of norms relative to the largest column: the product of two
            // squared norms itself underflows below 1e-11, columns above the floor
            // do not; and in float32, the margin being 1e-3 -- a float64 root in
            // every warp is 1 us of a round.)
            int cnt = 0;
            bool met = split == 1;
            for (int P0 = 0; P0 < npairs; P0 += 32) {
                const int P = P0 + lane;
                bool work = false;
                int a = 0, c = 0;
                if (P < npairs) {
                    a = circle_item(P, r, nb);
                    c = circle_item(nb - 1 - P, r, nb);
                    const T a1 = __ldcg(ti + 2 * a), a2 = __ldcg(ti + 2 * a + 1);
                    const T c1 = __ldcg(ti + 2 * c), c2 = __ldcg(ti + 2 * c + 1);
                    const T n1 = a1 > c1 ? a1 : c1, n2 = a1 > c1 ? (a2 > c1 ? a2 : c1) : (c2 > a1 ? c2 : a1);
                    T other = n2;
                    if (!KEEP)
                        other = T(d.p) * cx.scale * (T)(sqrt_approx((float)(n1 * cx.inv_scale)) * sqrt_approx((float)(n2 * cx.inv_scale)));
                    work = !((n1 + other) * T(1.001) <= cx.tau * cx.tau) &&
                           !(n2 * T(4) <= cx.floor2);
                    if (!work && rank == 0 && warp == 0) {
                        to[2 * a] = a1; to[2 * a + 1] = a2;
                        to[2 * c] = c1; to[2 * c + 1] = c2;
                    }
                }
                unsigned mask = __ballot_sync(0xffffffffu, work);
                while (mask) {
                    const int bit = __ffs(mask) - 1;
                    mask &= mask - 1;
                    if (cnt++ % nteams != team) continue;
                    const int pa = __shfl_sync(0xffffffffu, a, bit), pc = __shfl_sync(0xffffffffu, c, bit);
                    mine = fmax(mine, osj_pivot<T, NT, KEEP>(sm, cl, cx, pa, pc, to + 2 * pa, to + 2 * pc));
                    met = true;
                    if (clusterless) cx.gpart = gparts + ((flip ^= 1) ? GP : 0);
                }
            }
            // a split pivot of a cluster has one cluster barrier inside; every CTA passes
            // exactly one per round (a round has at most one pivot per team)
            if (!met && !clusterless) cl.sync();
            sync_block();
            if (clusterless && sm.fail) break;
            par ^= 1;
        }
        if (t == 0) {
            atomic_max_nonneg(d.off + sw % 3, mine);
            if (rank == 0) d.off[(sw + 1) % 3] = T(0);
        }
        sync_block();
        if (clusterless && sm.fail) break;
        const T o = __ldcg(d.off + sw % 3);
        if (rank == 0 && t == 0 && sweeps_run) sweeps_run[mat] += 1;
        if (o <= t_eff || (quad_exit && T(16) * o * o <= t_eff)) break;
    }
    if (clusterless && t == 0) {
        // the last CTA to leave makes the workspace ready for the next launch
        if (sm.fail) *d.fail = 1;
        else if (atomicInc(head + 1, (unsigned)csize - 1) == (unsigned)csize - 1) {
            head[0] = 0;
            for (int i = 0; i < npairs; ++i) head[GRID_HEAD + i] = 0;
        }
    }
}

// pivots of a round
template <typename T>
int pairs_of(int p) { return (p + 2 * Cfg<T>::OB - 1) / (2 * Cfg<T>::OB); }

template <typename T>
size_t smem_bytes(const OsjShape& sh) {
    constexpr size_t B2 = Smem<T>::B2, part = Smem<T>::PART;
    size_t words = Smem<T>::STAGE;
    if (sh.wide) {
        const size_t w = B2 * (size_t)wpanel_stride<T>(sh.max_p, sh.split);
        // a tile may read (never write) up to three 32-row groups past the last one
        words = (sh.split > 1 ? part + w : std::max(part, w)) + B2 * (size_t)panel_stride<T>(sh.max_L, sh.split) + 128;
    }
    return sizeof(Smem<T>) + sizeof(T) * words;
}

template <typename T, int NT, bool KEEP>
cudaError_t launch(const OsjDesc<T>* d_desc, int nmat, OsjShape shape, int sweeps, T tol, int* sweeps_run,
                   cudaStream_t s, int quad_exit, const int* list, int* resident) {
    // resident != nullptr: no launch, only how many such clusters fit the device
    static std::atomic<uint64_t> smem_set{0};
    cudaError_t e = ensure_smem_limit(osj_svd<T, NT, KEEP>, NT == NT_FEW ? (int)SMEM_MAX : (int)smem_bytes<T>(OsjShape{1, 1, 0, 1, 1, 0}),
                                      smem_set);
    if (e != cudaSuccess) return e;
    if (!shape.grid && shape.cluster > 8) {
        e = cudaFuncSetAttribute(osj_svd<T, NT, KEEP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    const bool clusterless = shape.grid != 0;
    if (clusterless && resident) {
        int dev = 0, sms = 0, per_sm = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, osj_svd<T, NT, KEEP>, NT, smem_bytes<T>(shape));
        *resident = per_sm * sms / shape.cluster;
        return e;
    }
    cfg.gridDim = dim3((unsigned)shape.cluster, (unsigned)nmat, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes<T>(shape);
    cfg.stream = s;
    cudaLaunchAttribute at;
    if (clusterless) {
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
    } else {
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)shape.cluster; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    }
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (resident) return cudaOccupancyMaxActiveClusters(resident, osj_svd<T, NT, KEEP>, &cfg);
    e = cudaLaunchKernelEx(&cfg, osj_svd<T, NT, KEEP>, d_desc, sweeps, tol, sweeps_run, quad_exit, shape.split, shape.grid, list);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// blocks of this shape that fit the current device at once; the runtime's
// answer (some 10 us a query, and a shape is chosen by a dozen) is kept per
// device, cluster size, thread count and shared memory
template <typename T>
int resident_clusters(const OsjShape& sh) {
    const size_t smem = smem_bytes<T>(sh);
    if (smem > SMEM_MAX) return 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, size_t>, int> known;
    const auto key = std::make_tuple(dev, sh.cluster, sh.wide + 2 * sh.grid, smem);
    {
        std::lock_guard<std::mutex> lock(mu);
        const auto it = known.find(key);
        if (it != known.end()) return it->second;
    }
    int n = 0;
    // (both schedules use the same shared memory and register limits)
    const cudaError_t e = sh.wide ? launch<T, NT_FEW, false>(nullptr, 1, sh, 0, T(0), nullptr, nullptr, 0, nullptr, &n)
                                  : launch<T, NT_MANY, false>(nullptr, 1, sh, 0, T(0), nullptr, nullptr, 0, nullptr, &n);
    if (e != cudaSuccess) n = 0;
    (void)cudaGetLastError();
    std::lock_guard<std::mutex> lock(mu);
    if (known.size() > 4096) known.clear();
    known[key] = n;
    return n;
}

}  // namespace

template <typename T>
int osj_max_cluster() {
    // 16 (the non-portable limit) when the device schedules clusters that
    // large for this kernel, else 8
    static std::atomic<int> big_ok{-1};
    if (big_ok.load() < 0) big_ok.store(resident_clusters<T>(OsjShape{16, 1, 0, 1, 1, 0}) > 0 ? 1 : 0);
    return big_ok.load() ? 16 : 8;
}

template <typename T>
size_t osj_grid_head(int p) { return sizeof(unsigned) * grid_head_words(pairs_of<T>(p)); }
template <typename T>
size_t osj_grid_bytes(int p) {
    return osj_grid_head<T>(p) + sizeof(T) * (size_t)pairs_of<T>(p) * 2 * Smem<T>::PART;
}

template <typename T>
OsjShape osj_shape(int nmat, int max_p, int max_L, int cluster, bool grid, int together) {
    // Cluster size: the caller's choice (autotuned), else the largest (up to
    // one CTA per pivot of a round) at which every block's cluster can be
    // resident at once -- a block waiting for a second wave would double the
    // time of the whole batch.  A cluster with room for several CTAs per pivot
    // splits its pivots, while a member keeps at least two chunks of rows.
    // Wide CTAs are taken while that leaves at most twice as many pivots to a
    // CTA as the streamed form would: ten blocks of 11 pivots fit as clusters of
    // 10 wide or 11 streamed CTAs, 170 against 225 ms over the 245 iterations of
    // the 500 x 5000 solve; 12 blocks of 13 pivots as 10 or 13, 188 against 266
    // (6 wide, 249); 40 blocks of 18 pivots as 3 or 10, 2.9 against 2.0 s.
    const int pairs = std::max(1, pairs_of<T>(max_p)), cmax = osj_max_cluster<T>();
    const int limit = cluster > 0 ? std::min(cluster, cmax) : cmax;
    auto fits = [&](const OsjShape& sh) { return resident_clusters<T>(sh) >= nmat; };
    auto in_cluster = [&]() {
    for (int split = 4; split > 1; split /= 2) {
        const OsjShape sh{pairs * split, split, 1, max_L, max_p, 0};
        if (sh.cluster <= limit && split * 64 <= max_L + max_p && fits(sh)) return sh;
    }
    // the largest cluster of each form
    auto largest = [&](int wide) {
        for (int c = std::min(limit, pairs); c > 0; --c) {
            const OsjShape sh{c, 1, wide, max_L, max_p, 0};
            if (fits(sh) || (!wide && cluster > 0)) return sh;
        }
        return OsjShape{wide ? 0 : 1, 1, wide, max_L, max_p, 0};
    };
    const OsjShape wide = largest(1), streamed = largest(0);
    if (wide.cluster > 0 && ceil_div(pairs, wide.cluster) <= 2 * ceil_div(pairs, streamed.cluster)) return wide;
    return streamed;
    };
    OsjShape best = in_cluster();
    if (!grid || cluster > 0) return best;
    // Without a cluster the CTAs of a block may lie anywhere, and there may be more
    // than 16.  The estimate, in us a round: a pivot takes about 17 whatever its
    // size (measure, inner rotations, R) and its Gram and update by the rate
    // measured on one SM, over the CTAs that share it; a meeting through memory
    // costs 2 to 3 more than a cluster barrier, and a split pivot has one inside.
    // (Whole pivots gain nothing: 10 blocks of 11, as clusters of 10 or so, 172 and
    // 175 ms in the 500 x 5000 solve.)  The 1000 x 487 float32 SVT, 64 CTAs for 16,
    // went from 16.5 to 12 ms; the 100 x 500 float64 one, 112 for 14, from 8 to 4.
    const double b2 = 2.0 * Cfg<T>::OB, work = (2.0 * max_L + max_p) * b2 * b2 / (sizeof(T) == 4 ? 110e3 : 3.7e3);
    auto cost = [&](const OsjShape& sh) {
        const int turns = (int)ceil_div((int64_t)pairs * sh.split, sh.cluster);
        return turns * (17.0 + work / sh.split) * (sh.wide ? 1.0 : 2.0) + (sh.grid ? 5.0 : 0.0);
    };
    // Its CTAs are all resident or none, so launches that do not fit beside one
    // another run in turn: each gets its share of the device.  (Eight threads with
    // SVTs of 100 x 500 float64: 30 ms a call when each launch takes 112 CTAs, 8.7
    // in clusters of 14; four threads 15 and, of 28 CTAs each, 5.5; of 1000 x 487
    // float32 46 and 21, 29 and 14.)  Whole solves are not counted: eight at once
    // are bound by their setup and the host's launches, and gain by what the form
    // saves each (float64 100 x 200: 330 ms with it, 399 without).
    auto consider = [&](const OsjShape& sh) {
        if (resident_clusters<T>(sh) >= nmat * together && cost(sh) < cost(best)) best = sh;
    };
    for (int split = Cfg<T>::NSLOT; split > 1; split /= 2) consider({pairs * split, split, 1, max_L, max_p, 1});
    return best;
}

namespace {
std::atomic<int> g_jacobi_calls[64];       // per device
}
JacobiCall::JacobiCall() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
    slot = dev & 63;
    g_jacobi_calls[slot].fetch_add(1, std::memory_order_relaxed);
}
JacobiCall::~JacobiCall() { g_jacobi_calls[slot].fetch_sub(1, std::memory_order_relaxed); }
int JacobiCall::together() const { return std::max(1, g_jacobi_calls[slot].load(std::memory_order_relaxed)); }

template <typename T>
cudaError_t osj_sweeps(const OsjDesc<T>* d_desc, int nmat, OsjShape shape, int sweeps, T tol, int* sweeps_run,
                       cudaStream_t s, OsjMode mode, int quad_exit, const int* list) {
    if (nmat <= 0 || sweeps <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 4) {
        if (mode == OsjMode::kept)
            return shape.wide ? launch<T, NT_FEW, true>(d_desc, nmat, shape, sweeps, tol, sweeps_run, s, quad_exit, list, nullptr)
                              : launch<T, NT_MANY, true>(d_desc, nmat, shape, sweeps, tol, sweeps_run, s, quad_exit, list, nullptr);
    }
    return shape.wide ? launch<T, NT_FEW, false>(d_desc, nmat, shape, sweeps, tol, sweeps_run, s, quad_exit, list, nullptr)
                      : launch<T, NT_MANY, false>(d_desc, nmat, shape, sweeps, tol, sweeps_run, s, quad_exit, list, nullptr);
}

template cudaError_t osj_sweeps<float>(const OsjDesc<float>*, int, OsjShape, int, float, int*, cudaStream_t, OsjMode, int, const int*);
template cudaError_t osj_sweeps<double>(const OsjDesc<double>*, int, OsjShape, int, double, int*, cudaStream_t, OsjMode, int, const int*);
template OsjShape osj_shape<float>(int, int, int, int, bool, int);
template OsjShape osj_shape<double>(int, int, int, int, bool, int);
template size_t osj_grid_head<float>(int);
template size_t osj_grid_head<double>(int);
template size_t osj_grid_bytes<float>(int);
template size_t osj_grid_bytes<double>(int);
template int osj_max_cluster<float>();
template int osj_max_cluster<double>();

}  // namespace lrr

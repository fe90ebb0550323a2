// Multi right-hand-side solve: k systems A x_c = b_c (c < k <= 32) sharing
// one hierarchy, advanced together (arxiv 2210.16660, Sec. 3.1 / Sec. 5 per
// column; the hierarchy is built once and reused, Sec. 2 / Sec. 4).
//
// Every vector is an n x K row-major block (the K values of a row are
// contiguous; K = k rounded up to a power of two, at least 4, padding
// columns are zero and inactive). One thread per (row, column): the K threads of a row read
// the same matrix entry (one broadcast load) and K consecutive vector values
// (one coalesced load), so each stored entry is read once per sweep for all
// columns (SpMM). Each column keeps its own Krylov scalars, iteration count,
// residual history and status; a column that has converged or failed stops
// changing (alpha = 0) while the others go on. Same V-cycle structure and
// reading of the method as the single right-hand-side path.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "internal.cuh"
#include "reduce.cuh"
#include "sell_row.cuh"

namespace pcgamg {

namespace {

constexpr int kMB = 256;         // threads per block
constexpr int kMaxK = 32;

template <typename T>
__device__ __forceinline__ T ldg(const T *p) { return __ldg(p); }

// Each thread owns V consecutive columns of one row (one 16-byte vector: 4
// floats or 2 doubles), so a row takes K / V threads, a warp covers 32V/K
// consecutive rows, a neighbour row's column group is one vector load, and
// the matrix entry of a row is one broadcast load shared by its threads.
template <typename T>
struct VW {
    static constexpr int V = 16 / (int)sizeof(T);
};

template <typename T, int V>
__device__ __forceinline__ void ld_vec(const T *p, T (&o)[V]) {
    if constexpr (sizeof(T) == 4) {
        float4 u = __ldg(reinterpret_cast<const float4 *>(p));
        o[0] = u.x; o[1] = u.y; o[2] = u.z; o[3] = u.w;
    } else {
        double2 u = __ldg(reinterpret_cast<const double2 *>(p));
        o[0] = u.x; o[1] = u.y;
    }
}

template <typename T, int V>
__device__ __forceinline__ void ld_vec_cg(const T *p, T (&o)[V]) {
    if constexpr (sizeof(T) == 4) {
        float4 u = __ldcg(reinterpret_cast<const float4 *>(p));
        o[0] = u.x; o[1] = u.y; o[2] = u.z; o[3] = u.w;
    } else {
        double2 u = __ldcg(reinterpret_cast<const double2 *>(p));
        o[0] = u.x; o[1] = u.y;
    }
}

template <typename T, int V>
__device__ __forceinline__ void st_vec(T *p, const T (&o)[V]) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
        *reinterpret_cast<double2 *>(p) = make_double2(o[0], o[1]);
    }
}

// acc[v] += sum_k a_k x(j_k)[v] over one sliced-ELL row, entries in storage
// order; U entries' columns and values are loaded before their gathers (level
// 0, Gauss-Seidel: a second chunk in flight costs more in registers than it
// gains there).
template <int U, bool STREAM, int V, typename IDX, typename T, typename F>
__device__ __forceinline__ void sell_row_vec(const IDX *__restrict__ c, const T *__restrict__ a, int w, int row,
                                             F xvec, T (&acc)[V]) {
#pragma unroll
    for (int v = 0; v < V; v++) acc[v] = 0;
    int k = 0;
    for (; k + U <= w; k += U) {
        int j[U];
        T av[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            j[u] = col_of(ld_mat<STREAM>(c + 32 * (k + u)), row);
            av[u] = ld_mat<STREAM>(a + 32 * (k + u));
        }
        T x[U][V];
#pragma unroll
        for (int u = 0; u < U; u++) xvec(j[u], x[u]);
#pragma unroll
        for (int u = 0; u < U; u++)
#pragma unroll
            for (int v = 0; v < V; v++) acc[v] += av[u] * x[u][v];
    }
    for (; k < w; k++) {
        int j = col_of(ld_mat<STREAM>(c + 32 * k), row);
        T av = ld_mat<STREAM>(a + 32 * k);
        T x[V];
        xvec(j, x);
#pragma unroll
        for (int v = 0; v < V; v++) acc[v] += av * x[v];
    }
}

// Thread (row i, first column c0) of a K-column block; grid-stride over
// n * (K / V) threads.
#define MK_FOR(nrows, V)                                                                      \
    for (int64_t g_ = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;                         \
         g_ < (int64_t)(nrows) * (K / (V)); g_ += (int64_t)gridDim.x * blockDim.x)
#define MK_IDX(V)                                                                             \
    int i = (int)(g_ / (K / (V)));                                                            \
    int c0 = (int)(g_ % (K / (V))) * (V);                                                     \
    int64_t e0 = (int64_t)i * K + c0;

// The columns still iterating (run[c]) and whether the solve has ended (run[K]),
// read once per block: thread c loads run_flag() and share_run() hands it on.
// The state lies in a few sectors of L2, which serve one request after
// another: read by every thread, those requests were what the kernels with
// one row per thread waited for (k_prolong_m of 218,800 rows x 32 in float32
// 51.5 us, 14.3 so; k_restrict_m to it 55.0 and 27.8).
// Small levels' kernels load the flag before their gathers and share it only
// before the store.
template <int K>
__device__ __forceinline__ int run_flag(const CtlM *ctl) {
    const int c = threadIdx.x;
    return c < K ? __ldcg(&ctl->active[c]) : c == K ? __ldcg(&ctl->done) : 0;
}

template <int K>
__device__ __forceinline__ const int *share_run(int flag) {
    __shared__ int run[K + 1];
    if (threadIdx.x <= K) run[threadIdx.x] = flag;
    __syncthreads();
    return run;
}

// Whether any of the V columns from c0 is still iterating.
template <int V>
__device__ __forceinline__ bool group_live(const int *run, int c0) {
    int a = 0;
#pragma unroll
    for (int v = 0; v < V; v++) a |= run[c0 + v];
    return a != 0;
}

// First column of a thread's fixed column group.
#define MK_C0(V) ((int)((((int64_t)blockIdx.x * blockDim.x + threadIdx.x) % (K / (V))) * (V)))

// A thread's column group is fixed over its grid-stride loop (the stride is a
// multiple of K / V); a group whose columns have all stopped skips its rows,
// so a block with few live columns moves only their vectors. The arithmetic
// of a live column does not depend on which other columns are live.
#define MK_LIVE(V) const bool live_ = group_live<V>(run, MK_C0(V));

// Per-column sums of NV quantities: a thread holds a[s][v], the s-th quantity
// of column c0 + v (c0 fixed per thread). The block's values meet in shared
// memory by column and a warp adds one column at a time (reduce.cuh), so no
// warp pays a float64 shuffle tree per quantity and column. Writes the block's
// partials (layout [quantity][column][block]); true in every thread of the
// last block to finish.
template <int K, int V, int NV>
__device__ __forceinline__ bool publish_cols(double (&a)[NV][V], double *partials, unsigned *counter) {
    constexpr int TPR = K / V, R = kMB / TPR;  // threads per row, values per column
    __shared__ double sh[NV * K * R];
    __shared__ bool last;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = (int)(threadIdx.x % TPR) * V, r = threadIdx.x / TPR;
#pragma unroll
    for (int s = 0; s < NV; s++)
#pragma unroll
        for (int v = 0; v < V; v++) sh[(s * K + c0 + v) * R + r] = a[s][v];
    __syncthreads();
    const int G = gridDim.x;
    for (int q = w; q < NV * K; q += kMB / 32) {
        double t = lane < R ? sh[q * R + lane] : 0.0;
        for (int k = lane + 32; k < R; k += 32) t += sh[q * R + k];
        t = warp_sum(t);
        if (lane == 0) partials[(int64_t)q * G + blockIdx.x] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = atomicAdd(counter, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    return last;
}

// Last block: res[q] = sum over blocks of partials[q][.], q < NV K.
template <int K, int NV>
__device__ __forceinline__ void final_cols(const double *partials, double *res) {
    __threadfence();
    const int G = gridDim.x;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int q = w; q < NV * K; q += kMB / 32) {
        const double *src = partials + (int64_t)q * G;
        double t = 0.0;
        for (int k0 = lane; k0 < G; k0 += 32 * 8) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; u++) x[u] = k0 + 32 * u < G ? __ldcg(src + k0 + 32 * u) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; u++)
                if (k0 - lane + 32 * u < G) t += x[u];
        }
        t = warp_sum(t);
        if (lane == 0) res[q] = t;
    }
    __syncthreads();
}

__device__ __forceinline__ void col_fail(CtlM *c, int col, int status) {
    c->status[col] = status;
    c->active[col] = 0;
}

// Every thread of the last block: done once no column is active. Thread c < K
// passes column c's flag.
__device__ __forceinline__ void update_done(CtlM *c, int active) {
    const int any = __syncthreads_or(active);
    if (threadIdx.x == 0 && !any) c->done = 1;
}

// ------------------------------------------------------------ V-cycle
// Level 0 and the other large levels: t = p (b - A xpre). Five resident blocks
// per SM: more gathers in flight than the registers the compiler would take
// (96^3 x 32: solves 162.8 -> 159.6 ms; served burst 43.9 -> 42.6 ms).
template <typename T, typename IDX, int K, int U, bool STREAM>
__global__ void __launch_bounds__(kMB, 5) k_down_m(int n, const int32_t *__restrict__ sptr,
                                               const IDX *__restrict__ col, const T *__restrict__ val,
                                               const T *__restrict__ xpre, const T *__restrict__ b,
                                               const T *__restrict__ p, T *__restrict__ t,
                                               const CtlM *__restrict__ ctl) {
    constexpr int V = VW<T>::V;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    MK_LIVE(V)
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        int s = i >> 5, lane = i & 31;
        int32_t base = ldg(sptr + s);
        int w = (ldg(sptr + s + 1) - base) >> 5;
        T acc[V];
        sell_row_vec<U, STREAM, V>(col + base + lane, val + base + lane, w, i,
                                   [&](int j, T (&x)[V]) { ld_vec<T, V>(xpre + (int64_t)j * K + c0, x); }, acc);
        T bv[V], o[V];
        ld_vec<T, V>(b + e0, bv);
        T pi = ldg(p + i);
#pragma unroll
        for (int v = 0; v < V; v++) o[v] = pi * (bv[v] - acc[v]);
        st_vec<T, V>(t + e0, o);
    }
}

// k_down_m and k_post_m on the coarse levels, which wait for latency: one
// (row, column group) per thread, its first U entries and the weight loaded
// before the wait, the next chunk's entries in flight during the gathers.
template <typename T, typename IDX, int K, int U>
__global__ void __launch_bounds__(kMB) k_down_c(int n, const int32_t *__restrict__ sptr,
                                               const IDX *__restrict__ col, const T *__restrict__ val,
                                               const IDX *__restrict__ upat, const T *__restrict__ xpre,
                                               const T *__restrict__ b, const T *__restrict__ p, T *__restrict__ t,
                                               const CtlM *__restrict__ ctl) {
    constexpr int V = VW<T>::V;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(g / (K / V)), c0 = (int)(g % (K / V)) * V;
    const bool in = i < n;
    SellRow<U, false, IDX, T> R;
    T pi = 0;
    if (in) {
        R.load(sptr, col, val, i, upat);
        pi = ldg(p + i);
    }
    pdl_enter();
    xpre = after_wait(xpre);
    b = after_wait(b);
    ctl = after_wait(ctl);
    const int flag = run_flag<K>(ctl);
    const int64_t e0 = (int64_t)i * K + c0;
    T bv[V], acc[V], o[V] = {};
    if (in) {
        ld_vec<T, V>(b + e0, bv);
        R.template dot_vec<V>(i, [&](int j, T (&x)[V]) { ld_vec<T, V>(xpre + (int64_t)j * K + c0, x); }, acc);
#pragma unroll
        for (int v = 0; v < V; v++) o[v] = pi * (bv[v] - acc[v]);
    }
    const int *run = share_run<K>(flag);
    if (in && !run[K] && group_live<V>(run, c0)) st_vec<T, V>(t + e0, o);
}

template <typename T, typename IDX, int K, int U>
__global__ void __launch_bounds__(kMB) k_post_c(int n, const int32_t *__restrict__ sptr,
                                               const IDX *__restrict__ col, const T *__restrict__ val,
                                               const IDX *__restrict__ upat, const T *__restrict__ xp,
                                               const T *__restrict__ b, const T *__restrict__ dinv,
                                               T *__restrict__ z, const CtlM *__restrict__ ctl) {
    constexpr int V = VW<T>::V;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(g / (K / V)), c0 = (int)(g % (K / V)) * V;
    const bool in = i < n;
    SellRow<U, false, IDX, T> R;
    T d = 0;
    if (in) {
        R.load(sptr, col, val, i, upat);
        d = ldg(dinv + i);
    }
    pdl_enter();
    xp = after_wait(xp);
    b = after_wait(b);
    ctl = after_wait(ctl);
    const int flag = run_flag<K>(ctl);
    const int64_t e0 = (int64_t)i * K + c0;
    T xv[V], bv[V], acc[V], o[V] = {};
    if (in) {
        ld_vec<T, V>(xp + e0, xv);
        ld_vec<T, V>(b + e0, bv);
        R.template dot_vec<V>(i, [&](int j, T (&x)[V]) { ld_vec<T, V>(xp + (int64_t)j * K + c0, x); }, acc);
#pragma unroll
        for (int v = 0; v < V; v++) o[v] = xv[v] + d * (bv[v] - acc[v]);
    }
    const int *run = share_run<K>(flag);
    if (in && !run[K] && group_live<V>(run, c0)) st_vec<T, V>(z + e0, o);
}

// b_c[I] = sum of t over the members of aggregate I in index order (and
// xpre_c = dinv_c b_c), one (coarse row, column group) per thread; the first
// four members are static and read before the wait.
template <typename T, typename TO, bool PRE, int K>
__global__ void __launch_bounds__(kMB) k_restrict_m(int nc, const int32_t *__restrict__ rptr,
                                                   const int32_t *__restrict__ ridx, const T *__restrict__ t,
                                                   TO *__restrict__ bc, const T *__restrict__ dinvc,
                                                   T *__restrict__ xprec, const CtlM *__restrict__ ctl) {
    constexpr int V = VW<T>::V, M = 4;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(g / (K / V)), c0 = (int)(g % (K / V)) * V;
    const bool in = i < nc;
    int32_t q0 = 0, q1 = 0;
    int m[M];
    T d = 0;
    if (in) {
        q0 = ldg(rptr + i);
        q1 = ldg(rptr + i + 1);
#pragma unroll
        for (int u = 0; u < M; u++) m[u] = q0 + u < q1 ? ldg(ridx + q0 + u) : 0;
        if (PRE) d = ldg(dinvc + i);
    }
    pdl_enter();
    t = after_wait(t);
    ctl = after_wait(ctl);
    const int flag = run_flag<K>(ctl);
    const int64_t e0 = (int64_t)i * K + c0;
    T s[V], x[M][V];
#pragma unroll
    for (int v = 0; v < V; v++) s[v] = 0;
#pragma unroll
    for (int u = 0; u < M; u++)
        if (q0 + u < q1) ld_vec<T, V>(t + (int64_t)m[u] * K + c0, x[u]);
#pragma unroll
    for (int u = 0; u < M; u++)
        if (q0 + u < q1) {
#pragma unroll
            for (int v = 0; v < V; v++) s[v] += x[u][v];
        }
    for (int32_t q = q0 + M; q < q1; q++) {
        T y[V];
        ld_vec<T, V>(t + (int64_t)ldg(ridx + q) * K + c0, y);
#pragma unroll
        for (int v = 0; v < V; v++) s[v] += y[v];
    }
    const int *run = share_run<K>(flag);
    if (!in || run[K] || !group_live<V>(run, c0)) return;
#pragma unroll
    for (int v = 0; v < V; v++) bc[e0 + v] = (TO)s[v];
    if (PRE) {
        T o[V];
#pragma unroll
        for (int v = 0; v < V; v++) o[v] = d * s[v];
        st_vec<T, V>(xprec + e0, o);
    }
}

// x = B b for K columns on the directly solved level (float64): the coarsest
// inverse, or the explicit operator of the small levels (amg_hier::op). One
// warp per (row, pair of columns), lanes striding over the row with coalesced
// loads, then the warp's sum.
template <typename TO, int K>
__global__ void __launch_bounds__(kMB) k_coarse_m(int nL, const double *__restrict__ ainv,
                                                 const double *__restrict__ bL, TO *__restrict__ xL,
                                                 const CtlM *__restrict__ ctl) {
    constexpr int V = 2;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    int warp = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (warp >= nL * (K / V)) return;  // whole warps
    int row = warp / (K / V), c0 = (warp % (K / V)) * V;
    if (!group_live<V>(run, c0)) return;
    const double *a = ainv + (int64_t)row * nL;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
    for (int j = lane; j < nL; j += 32) {
        double aj = ldg(a + j);
        double2 bj = __ldg(reinterpret_cast<const double2 *>(bL + (int64_t)j * K + c0));
        s0 += aj * bj.x;
        s1 += aj * bj.y;
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (lane == 0) {
        xL[(int64_t)row * K + c0] = (TO)s0;
        xL[(int64_t)row * K + c0 + 1] = (TO)s1;
    }
}

template <typename T, int K>
__global__ void __launch_bounds__(kMB) k_prolong_m(int n, const T *__restrict__ xpre, const T *__restrict__ p,
                                                  const int32_t *__restrict__ agg, const T *__restrict__ xc,
                                                  T *__restrict__ xp, const CtlM *__restrict__ ctl) {
    constexpr int V = VW<T>::V;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    MK_LIVE(V)
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        T x[V];
        ld_vec<T, V>(xpre + e0, x);
        int a = ldg(agg + i);
        if (a >= 0) {
            T pi = ldg(p + i), y[V];
            ld_vec<T, V>(xc + (int64_t)a * K + c0, y);
#pragma unroll
            for (int v = 0; v < V; v++) x[v] += pi * y[v];
        }
        st_vec<T, V>(xp + e0, x);
    }
}

// Per-column rho = r.z and beta (see the single-column k_axpy_p) from the
// threads' sums of r.z and, with NV = 2, z.q_old.
template <int K, int V, int NV>
__device__ __forceinline__ void finish_rho_m(double (&sums)[NV][V], double *partials, CtlM *ctl) {
    __shared__ double res[NV * K];
    if (!publish_cols<K, V, NV>(sums, partials, &ctl->counter[0])) return;
    final_cols<K, NV>(partials, res);
    if (threadIdx.x == 0) ctl->counter[0] = 0;
    const int c = threadIdx.x;
    if (c < K && __ldcg(&ctl->active[c])) {
        const double rho = res[c], zqc = NV == 2 ? res[(NV - 1) * K + c] : 0.0;
        if (!isfinite(rho) || !isfinite(zqc)) {
            col_fail(ctl, c, AMG_ERR_NAN);
        } else if (!(rho > 0.0)) {
            col_fail(ctl, c, AMG_ERR_BREAKDOWN);
        } else {
            ctl->rho[c] = rho;
            double beta = 0.0;
            if (!__ldcg(&ctl->restart[c]))
                beta = NV == 2 ? -zqc / __ldcg(&ctl->pq_old[c]) : rho / __ldcg(&ctl->rho_old[c]);
            ctl->beta[c] = beta;
        }
    }
}

// z = xp + D^-1 (b - A xp); DOT on level 0: per-column r.z and z.q_old, and
// the last block forms rho_c and beta_c. Below 16 columns four blocks per SM
// (registers for the row's gathers): served burst 43.9 -> 42.4 ms, 40^3 x 5
// 6.78 -> 6.68 ms.
template <typename T, typename TZ, bool DOT, bool FCG, typename IDX, int K, int U, bool STREAM>
__global__ void __launch_bounds__(kMB, K >= 16 ? 0 : 4) k_post_m(int n, const int32_t *__restrict__ sptr,
                                               const IDX *__restrict__ col, const T *__restrict__ val,
                                               const T *__restrict__ xp, const T *__restrict__ b,
                                               const T *__restrict__ dinv, TZ *__restrict__ z,
                                               const double *__restrict__ r64, const double *__restrict__ qold,
                                               double *partials, CtlM *ctl) {
    constexpr int V = VW<T>::V;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    constexpr int NV = FCG ? 2 : 1;
    double sums[NV][V] = {};
    MK_LIVE(V)
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        int s = i >> 5, lane = i & 31;
        int32_t base = ldg(sptr + s);
        int w = (ldg(sptr + s + 1) - base) >> 5;
        T acc[V];
        sell_row_vec<U, STREAM, V>(col + base + lane, val + base + lane, w, i,
                                   [&](int j, T (&x)[V]) { ld_vec<T, V>(xp + (int64_t)j * K + c0, x); }, acc);
        T xv[V], bv[V];
        ld_vec<T, V>(xp + e0, xv);
        ld_vec<T, V>(b + e0, bv);
        T d = ldg(dinv + i);
#pragma unroll
        for (int v = 0; v < V; v++) {
            const TZ zo = (TZ)(xv[v] + d * (bv[v] - acc[v]));
            z[e0 + v] = zo;
            if (DOT) {
                sums[0][v] += ldg(r64 + e0 + v) * (double)zo;
                if (FCG) sums[NV - 1][v] += (double)zo * ldg(qold + e0 + v);
            }
        }
    }
    if constexpr (DOT) finish_rho_m<K, V, NV>(sums, partials, ctl);
}

// ------------------------------------------------------------ hybrid Gauss-Seidel
// One sweep of the l1 hybrid Gauss-Seidel smoother for K columns (the
// single-column k_gs_warp per column group): one warp per (32-row slice,
// group of V columns), a lane per row. Phase one sums each row's entries with
// x_old except the in-block ones this pass has already updated; phase two
// runs the slice's rows in pass order in 32 steps, each finished value
// broadcast by a shuffle and added by the rows whose next in-block entry (in
// pass order) is that row. Needs blocks whose size divides 32 and rows with
// at most kGsPartM in-block entries of the pass.
constexpr int kGsPartM = 8;

template <typename T, typename IDX, int U, bool FWD, bool ZERO, bool STREAM, int K>
__global__ void __launch_bounds__(kMB) k_gs_warp_m(int n, int nb, int w, const int32_t *__restrict__ sptr,
                                                  const IDX *__restrict__ col, const T *__restrict__ val,
                                                  const int32_t *__restrict__ pci, const T *__restrict__ pv,
                                                  const T *__restrict__ dinv, const T *__restrict__ b,
                                                  const T *__restrict__ xo, T *__restrict__ xn,
                                                  const CtlM *__restrict__ ctl) {
    constexpr int V = VW<T>::V;
    constexpr int G = K / V;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    const int lane = threadIdx.x & 31;
    const int nsl = (n + 31) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t wi = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; wi < (int64_t)nsl * G; wi += nw) {
        const int sl = (int)(wi / G), c0 = (int)(wi % G) * V;
        if (!group_live<V>(run, c0)) continue;  // uniform over the warp
        const int i = (sl << 5) + lane;
        const bool valid = i < n;
        const int64_t e0 = (int64_t)i * K + c0;
        T acc[V];
#pragma unroll
        for (int v = 0; v < V; v++) acc[v] = 0;
        if (!ZERO && valid) {
            const int lo = (i / nb) * nb, hi = min(n, lo + nb);
            int32_t base = ldg(sptr + sl);
            int wd = (ldg(sptr + sl + 1) - base) >> 5;
            sell_row_vec<U, STREAM, V>(col + base + lane, val + base + lane, wd, i,
                                       [&](int j, T (&x)[V]) {
                                           bool done = FWD ? (j >= lo && j < i) : (j > i && j < hi);
                                           if (done) {
#pragma unroll
                                               for (int v = 0; v < V; v++) x[v] = 0;
                                           } else {
                                               ld_vec<T, V>(xo + (int64_t)j * K + c0, x);
                                           }
                                       },
                                       acc);
        }
        int rj[kGsPartM];
        T ra[kGsPartM];
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < kGsPartM; k++) {
            bool ok = valid && k < w;
            rj[k] = ok ? ldg(pci + (int64_t)i * w + k) : -1;
            ra[k] = ok ? ldg(pv + (int64_t)i * w + k) : T(0);
            cnt += rj[k] >= 0 ? 1 : 0;
        }
        int pj[kGsPartM];
        T pa[kGsPartM];
#pragma unroll
        for (int k = 0; k < kGsPartM; k++) {
            if (FWD) {
                pj[k] = rj[k];
                pa[k] = ra[k];
            } else {
                pj[k] = -1;
                pa[k] = T(0);
#pragma unroll
                for (int m = 0; m < kGsPartM; m++)
                    if (m == cnt - 1 - k) {
                        pj[k] = rj[m];
                        pa[k] = ra[m];
                    }
            }
        }
        T bv[V], xold[V], x[V];
        const T di = valid ? ldg(dinv + i) : T(0);
#pragma unroll
        for (int v = 0; v < V; v++) bv[v] = xold[v] = x[v] = 0;
        if (valid) {
            ld_vec<T, V>(b + e0, bv);
            if (!ZERO) ld_vec<T, V>(xo + e0, xold);
        }
#pragma unroll 2
        for (int step = 0; step < 32; step++) {
            const int t = FWD ? step : 31 - step;
            if (lane == t)
#pragma unroll
                for (int v = 0; v < V; v++) x[v] = ZERO ? di * (bv[v] - acc[v]) : xold[v] + di * (bv[v] - acc[v]);
            T xt[V];
#pragma unroll
            for (int v = 0; v < V; v++) xt[v] = __shfl_sync(0xffffffffu, x[v], t);
            if (pj[0] == (sl << 5) + t) {
#pragma unroll
                for (int v = 0; v < V; v++) acc[v] += pa[0] * xt[v];
#pragma unroll
                for (int k = 0; k + 1 < kGsPartM; k++) {
                    pj[k] = pj[k + 1];
                    pa[k] = pa[k + 1];
                }
                pj[kGsPartM - 1] = -1;
            }
        }
        if (valid) st_vec<T, V>(xn + e0, x);
    }
}

// Level 0 after the Gauss-Seidel post-smoothing: z = x (widened), r.z and
// (FCG) z.q_old per column; the last block forms rho and beta per column.
template <typename T, bool FCG, int K>
__global__ void __launch_bounds__(kMB) k_gs_finish0_m(int n, const T *__restrict__ x, const double *__restrict__ r64,
                                                     const double *__restrict__ qold, double *__restrict__ z,
                                                     double *partials, CtlM *ctl) {
    constexpr int V = VW<T>::V;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    constexpr int NV = FCG ? 2 : 1;
    double sums[NV][V] = {};
    MK_LIVE(V)
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        T xv[V];
        ld_vec<T, V>(x + e0, xv);
#pragma unroll
        for (int v = 0; v < V; v++) {
            double zo = (double)xv[v];
            z[e0 + v] = zo;
            sums[0][v] += ldg(r64 + e0 + v) * zo;
            if (FCG) sums[NV - 1][v] += zo * ldg(qold + e0 + v);
        }
    }
    finish_rho_m<K, V, NV>(sums, partials, ctl);
}

// ------------------------------------------------------------ Krylov
template <int K>
__global__ void __launch_bounds__(kMB) k_axpy_m(int n, const double *__restrict__ z, double *__restrict__ p,
                                               const CtlM *__restrict__ ctl) {
    constexpr int V = 2;
    pdl_enter();
    __shared__ double sbeta[K];
    if (threadIdx.x < K) sbeta[threadIdx.x] = __ldcg(&ctl->beta[threadIdx.x]);
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    MK_LIVE(V)
    int act[V];
    double beta[V];
#pragma unroll
    for (int v = 0; v < V; v++) {
        act[v] = run[MK_C0(V) + v];
        beta[v] = sbeta[MK_C0(V) + v];
    }
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        double zv[V], pv[V], o[V];
        ld_vec<double, V>(z + e0, zv);
        ld_vec_cg<double, V>(p + e0, pv);
#pragma unroll
        for (int v = 0; v < V; v++) o[v] = act[v] ? zv[v] + beta[v] * pv[v] : 0.0;
        st_vec<double, V>(p + e0, o);
    }
}

// Bound by the float64 pipe (two FMAs per entry and thread); from 16 columns on
// a full SM of warps at 32 registers, of which 84 bytes a thread are spilled,
// keeps it busier than fewer with more (96^3 x 32 mixed: whole solves 164 ms,
// 172 at the compiler's registers; 96^3 x 32 and 160^3 x 32 float64 308.4 and
// 1,644 ms, 315.5 and 1,683; 40^3 x 8 lost, 7.0 -> 7.3 ms, and 96^3 x 8 mixed
// with six blocks per SM too, 41.3 -> 43.2, so four below 16 columns).
template <typename IDX, int K>
__global__ void __launch_bounds__(kMB, K >= 16 ? 8 : 4) k_spmm_m(int n, const int32_t *__restrict__ sptr,
                                               const IDX *__restrict__ col, const double *__restrict__ val,
                                               const double *__restrict__ p, double *__restrict__ q,
                                               double *partials, CtlM *ctl) {
    constexpr int V = 2;
    pdl_enter();
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    double pq[1][V] = {};
    MK_LIVE(V)
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        int s = i >> 5, lane = i & 31;
        int32_t base = ldg(sptr + s);
        int w = (ldg(sptr + s + 1) - base) >> 5;
        double acc[V];
        sell_row_vec<kUnroll, true, V>(col + base + lane, val + base + lane, w, i,
                                       [&](int j, double (&x)[V]) { ld_vec<double, V>(p + (int64_t)j * K + c0, x); },
                                       acc);
        st_vec<double, V>(q + e0, acc);
        double pv[V];
        ld_vec<double, V>(p + e0, pv);
#pragma unroll
        for (int v = 0; v < V; v++) pq[0][v] += pv[v] * acc[v];
    }
    __shared__ double res[K];
    if (publish_cols<K, V, 1>(pq, partials, &ctl->counter[1])) {
        final_cols<K, 1>(partials, res);
        if (threadIdx.x == 0) ctl->counter[1] = 0;
        int c = threadIdx.x;
        if (c < K) {
            double alpha = 0.0;
            if (__ldcg(&ctl->active[c])) {
                double a = res[c];
                if (!isfinite(a)) col_fail(ctl, c, AMG_ERR_NAN);
                else if (!(a > 0.0)) col_fail(ctl, c, AMG_ERR_BREAKDOWN);
                else {
                    ctl->pq[c] = a;
                    alpha = __ldcg(&ctl->rho[c]) / a;
                }
            }
            ctl->alpha[c] = alpha;
        }
    }
}

// The mode's copy of r for the V-cycle, two columns at a time.
template <int MODE>
__device__ __forceinline__ void emit_r_m(int64_t e, int i, const double (&ri)[2], float *r32, const float *dinv32,
                                         float *xpre32, const double *dinv64, double *xpre64) {
    if (MODE == AMG_MODE_FCG32) {
        float d = __ldg(dinv32 + i);
        float a = (float)ri[0], b = (float)ri[1];
        *reinterpret_cast<float2 *>(r32 + e) = make_float2(a, b);
        *reinterpret_cast<float2 *>(xpre32 + e) = make_float2(d * a, d * b);
    } else {
        double d = __ldg(dinv64 + i);
        *reinterpret_cast<double2 *>(xpre64 + e) = make_double2(d * ri[0], d * ri[1]);
    }
}

template <int MODE, int K>
__global__ void __launch_bounds__(kMB) k_update_m(int n, const double *__restrict__ p,
                                                 const double *__restrict__ q, double *__restrict__ x,
                                                 double *__restrict__ r, float *__restrict__ r32,
                                                 const float *__restrict__ dinv32, float *__restrict__ xpre32,
                                                 const double *__restrict__ dinv64, double *__restrict__ xpre64,
                                                 double *partials, CtlM *ctl, double *hist, int hstride) {
    constexpr int V = 2;
    pdl_enter();
    __shared__ double salpha[K];
    if (threadIdx.x < K) salpha[threadIdx.x] = __ldcg(&ctl->alpha[threadIdx.x]);
    const int *run = share_run<K>(run_flag<K>(ctl));
    if (run[K]) return;
    double rr[1][V] = {};
    MK_LIVE(V)
    int act[V];
    double al[V];
#pragma unroll
    for (int v = 0; v < V; v++) {
        act[v] = run[MK_C0(V) + v];
        al[v] = salpha[MK_C0(V) + v];
    }
    MK_FOR(live_ ? n : 0, V) {
        MK_IDX(V)
        double rv[V], xv[V], pv[V], qv[V];
        ld_vec_cg<double, V>(r + e0, rv);
        ld_vec_cg<double, V>(x + e0, xv);
        ld_vec<double, V>(p + e0, pv);
        ld_vec<double, V>(q + e0, qv);
#pragma unroll
        for (int v = 0; v < V; v++) {
            if (act[v]) {
                xv[v] = xv[v] + al[v] * pv[v];
                rv[v] = rv[v] - al[v] * qv[v];
                rr[0][v] += rv[v] * rv[v];
            }
        }
        st_vec<double, V>(x + e0, xv);
        st_vec<double, V>(r + e0, rv);
        emit_r_m<MODE>(e0, i, rv, r32, dinv32, xpre32, dinv64, xpre64);
    }
    __shared__ double res[K];
    if (publish_cols<K, V, 1>(rr, partials, &ctl->counter[2])) {
        final_cols<K, 1>(partials, res);
        // one thread per column: its scalars, then whether any goes on
        const int c = threadIdx.x;
        int active = 0, check = 0;
        if (c < K && __ldcg(&ctl->active[c])) {
            const int it = __ldcg(&ctl->iter[c]) + 1;
            const double rel = sqrt(res[c]) / __ldcg(&ctl->bnorm[c]);
            ctl->iter[c] = it;
            ctl->rel[c] = rel;
            hist[(int64_t)c * hstride + it] = rel;
            ctl->rho_old[c] = __ldcg(&ctl->rho[c]);
            ctl->pq_old[c] = __ldcg(&ctl->pq[c]);
            ctl->restart[c] = 0;
            active = 1;
            if (!isfinite(rel)) {
                col_fail(ctl, c, AMG_ERR_NAN);
                active = 0;
            } else if (rel <= __ldcg(&ctl->rtol)) {
                ctl->check[c] = 1;
                check = 1;
            } else if (it >= __ldcg(&ctl->maxit)) {
                col_fail(ctl, c, AMG_ERR_NOCONV);
                active = 0;
            }
        }
        const int any_check = __syncthreads_or(check);
        if (c == 0) {
            ctl->counter[2] = 0;
            ctl->iter_all = __ldcg(&ctl->iter_all) + 1;
            ctl->any_check = any_check;
        }
        update_done(ctl, active);
    }
}

// r = b - A x. INIT: the columns marked pending (a new right-hand side),
// plus ||b||; otherwise only the columns whose recursive residual met rtol.
// The other columns keep their r.
template <bool INIT, int MODE, typename IDX, int K>
__global__ void __launch_bounds__(kMB) k_residual_m(int n, const int32_t *__restrict__ sptr,
                                                   const IDX *__restrict__ col, const double *__restrict__ val,
                                                   const double *__restrict__ b, const double *__restrict__ x,
                                                   double *__restrict__ r, float *__restrict__ r32,
                                                   const float *__restrict__ dinv32, float *__restrict__ xpre32,
                                                   const double *__restrict__ dinv64, double *__restrict__ xpre64,
                                                   double *partials, CtlM *ctl, double *hist, int hstride) {
    constexpr int V = 2;
    pdl_enter();
    // as run_flag: the columns to form the residual of, and whether any is left to do
    __shared__ int uses[K + 1];
    if (threadIdx.x < K)
        uses[threadIdx.x] = INIT ? __ldcg(&ctl->pending[threadIdx.x]) : __ldcg(&ctl->check[threadIdx.x]);
    if (threadIdx.x == K) uses[K] = !__ldcg(&ctl->done) && (INIT || __ldcg(&ctl->any_check));
    __syncthreads();
    if (!uses[K]) return;
    constexpr int NV = INIT ? 2 : 1;
    double sums[NV][V] = {};
    const bool use0 = uses[MK_C0(V)] != 0, use1 = uses[MK_C0(V) + 1] != 0;
    MK_FOR(use0 || use1 ? n : 0, V) {
        MK_IDX(V)
        int s = i >> 5, lane = i & 31;
        int32_t base = ldg(sptr + s);
        int w = (ldg(sptr + s + 1) - base) >> 5;
        double acc[V];
        sell_row_vec<kUnroll, true, V>(col + base + lane, val + base + lane, w, i,
                                       [&](int j, double (&xx)[V]) { ld_vec<double, V>(x + (int64_t)j * K + c0, xx); },
                                       acc);
        double bv[V], rv[V];
        ld_vec<double, V>(b + e0, bv);
        ld_vec_cg<double, V>(r + e0, rv);
        if (use0) rv[0] = bv[0] - acc[0];
        if (use1) rv[1] = bv[1] - acc[1];
        st_vec<double, V>(r + e0, rv);
        emit_r_m<MODE>(e0, i, rv, r32, dinv32, xpre32, dinv64, xpre64);
        if (use0) sums[0][0] += rv[0] * rv[0];
        if (use1) sums[0][1] += rv[1] * rv[1];
        if (INIT) {
            if (use0) sums[NV - 1][0] += bv[0] * bv[0];
            if (use1) sums[NV - 1][1] += bv[1] * bv[1];
        }
    }
    __shared__ double res[NV * K];
    if (publish_cols<K, V, NV>(sums, partials, &ctl->counter[3])) {
        final_cols<K, NV>(partials, res);
        const int c = threadIdx.x;
        int active = 0;
        if (c < K) {
            active = __ldcg(&ctl->active[c]);
            if (INIT && __ldcg(&ctl->pending[c])) {
                const double bn = sqrt(res[(NV - 1) * K + c]);
                ctl->pending[c] = 0;
                ctl->bnorm[c] = bn;
                ctl->status[c] = AMG_OK;
                ctl->iter[c] = 0;
                ctl->check[c] = 0;
                active = 0;
                int status = AMG_OK;
                if (c < __ldcg(&ctl->k)) {
                    if (!isfinite(bn) || !isfinite(res[c])) {
                        status = AMG_ERR_NAN;
                    } else if (bn == 0.0) {
                        ctl->true_rel[c] = 0.0;
                        hist[(int64_t)c * hstride] = 0.0;
                    } else {
                        const double rel = sqrt(res[c]) / bn;
                        ctl->rel[c] = rel;
                        ctl->true_rel[c] = rel;
                        hist[(int64_t)c * hstride] = rel;
                        if (!(rel <= __ldcg(&ctl->rtol))) {
                            if (__ldcg(&ctl->maxit) <= 0) {
                                status = AMG_ERR_NOCONV;
                            } else {
                                active = 1;
                                ctl->restart[c] = 1;
                            }
                        }
                    }
                }
                ctl->active[c] = active;
                if (status != AMG_OK) ctl->status[c] = status;
            } else if (!INIT && __ldcg(&ctl->check[c])) {
                const double rel = sqrt(res[c]) / __ldcg(&ctl->bnorm[c]);
                const int it = __ldcg(&ctl->iter[c]);
                ctl->check[c] = 0;
                ctl->true_rel[c] = rel;
                active = 0;
                if (!isfinite(rel)) {
                    col_fail(ctl, c, AMG_ERR_NAN);
                } else if (rel <= __ldcg(&ctl->rtol)) {
                    ctl->active[c] = 0;
                    ctl->status[c] = AMG_OK;
                } else {
                    ctl->restart[c] = 1;
                    hist[(int64_t)c * hstride + it] = rel;
                    if (it >= __ldcg(&ctl->maxit)) col_fail(ctl, c, AMG_ERR_NOCONV);
                    else active = 1;
                }
            }
        }
        if (c == 0) {
            ctl->counter[3] = 0;
            ctl->any_check = 0;
        }
        update_done(ctl, active);
    }
}

__global__ void k_zero_m(double *a, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = 0.0;
}

// Copies between the caller's n x k block and the internal n x K block.
__global__ void k_pack(const double *__restrict__ src, int k, double *__restrict__ dst, int K, int64_t n) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n * K) return;
    int64_t i = g / K;
    int c = (int)(g % K);
    dst[g] = c < k ? src[i * k + c] : 0.0;
}

// Unpack; columns with b = 0 get x = 0.
__global__ void k_unpack(const double *__restrict__ src, int K, double *__restrict__ dst, int k, int64_t n,
                         const CtlM *__restrict__ ctl) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n * k) return;
    int64_t i = g / k;
    int c = (int)(g % k);
    dst[g] = ctl->bnorm[c] == 0.0 ? 0.0 : src[i * K + c];
}

__global__ void k_set_cond_m(cudaGraphConditionalHandle hc, CtlM *ctl, int count_body) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if (count_body) {
        int b = ctl->bodies + 1;
        ctl->bodies = b;
        if (!ctl->done && b > (ctl->maxit + 1) / 2 + 1) {
            for (int c = 0; c < ctl->K; c++)
                if (ctl->active[c]) col_fail(ctl, c, AMG_ERR_NOCONV);
            ctl->done = 1;
        }
    }
    cudaGraphSetConditional(hc, ctl->done ? 0u : 1u);
}

inline int grid_of(int64_t items) { return (int)((items + kMB - 1) / kMB); }

template <typename T>
struct MP;
template <>
struct MP<float> {
    static const float *val(const Level &l) { return l.S.v32; }
    static const float *dinv(const Level &l) { return l.dinv32; }
    static const float *p(const Level &l) { return l.p32; }
    static float *b(MultiLevel &m) { return m.b32; }
    static float *x(MultiLevel &m) { return m.x32; }
    static float *t(MultiLevel &m) { return m.t32; }
    static float *xpre(MultiLevel &m) { return m.xpre32; }
    static float *xp(MultiLevel &m) { return m.xp32; }
    static const float *part(const Level &l, int d) { return l.gs_v32[d]; }
};
template <>
struct MP<double> {
    static const double *val(const Level &l) { return l.S.v64; }
    static const double *dinv(const Level &l) { return l.dinv; }
    static const double *p(const Level &l) { return l.p; }
    static double *b(MultiLevel &m) { return m.b64; }
    static double *x(MultiLevel &m) { return m.x64; }
    static double *t(MultiLevel &m) { return m.t64; }
    static double *xpre(MultiLevel &m) { return m.xpre64; }
    static double *xp(MultiLevel &m) { return m.xp64; }
    static const double *part(const Level &l, int d) { return l.gs_v64[d]; }
};

#define WITH_COLS_M(S, BODY)                               \
    do {                                                   \
        if ((S).col16) {                                   \
            using IDX = int16_t;                           \
            const IDX *cols = (S).col16;                   \
            [[maybe_unused]] const IDX *pats = (S).upat16; \
            BODY;                                          \
        } else {                                           \
            using IDX = int32_t;                           \
            const IDX *cols = (S).col;                     \
            [[maybe_unused]] const IDX *pats = (S).upat;   \
            BODY;                                          \
        }                                                  \
    } while (0)

// gs_nu Gauss-Seidel sweeps of level l for K columns: pre-smoothing
// (forward, from zero, into the level's xpre) or post-smoothing (backward,
// from xp, into x); sweeps alternate between the target and t so the last
// writes the target.
template <typename T, int K>
void launch_gs_m(amg_hier *h, MultiWS &W, int l, bool pre, const T *b, T *target, cudaStream_t s) {
    using P = MP<T>;
    constexpr int V = VW<T>::V;
    Level &lv = h->lev[l];
    MultiLevel &mv = W.lev[l];
    const int n = lv.A.n, nu = h->gs_nu, nb = gs_rows(n, h->gs_blocks), d = pre ? 0 : 1;
    const int w = lv.gs_w[d];
    const int grid = grid_of((((int64_t)n + 31) / 32) * (K / V) * 32);
    const T *src = pre ? nullptr : (const T *)P::xp(mv);
    const bool big = n > kSmallRows;
    for (int sw = 1; sw <= nu; sw++) {
        T *dst = (nu - sw) % 2 == 0 ? target : P::t(mv);
        const bool zero = pre && sw == 1;
#define PCG_GSM_LAUNCH(UU, FWD, ZERO, ST)                                                                        \
    WITH_COLS_M(lv.S, (launch_k(h->pdl, k_gs_warp_m<T, IDX, UU, FWD, ZERO, ST, K>, grid, kMB, s, n, nb, w,      \
                                lv.S.sptr, cols, P::val(lv), lv.gs_ci[d], P::part(lv, d), P::dinv(lv), b, src,  \
                                dst, W.ctl)))
#define PCG_GSM(UU, ST)                                  \
    do {                                                 \
        if (zero) PCG_GSM_LAUNCH(UU, true, true, ST);    \
        else if (pre) PCG_GSM_LAUNCH(UU, true, false, ST); \
        else PCG_GSM_LAUNCH(UU, false, false, ST);       \
    } while (0)
        if (l == 0) PCG_GSM(kUnroll, true);
        else if (big) PCG_GSM(kUnroll, false);
        else PCG_GSM(kUnrollSmall, false);
#undef PCG_GSM_LAUNCH
#undef PCG_GSM
        src = dst;
    }
}

// The level that K columns solve directly: the explicit operator of the first
// level whose product stays under kOpWorkM float64 FMAs (9 million take 14 us;
// at 8 columns a 992-row level's sweeps, transfers and coarse solve took 25),
// else the coarsest one.
constexpr int64_t kOpWorkM = 9000000;
int direct_level_m(const amg_hier *h, int K) {
    const int L = (int)h->lev.size() - 1;
    for (int l = h->op_first; l && l < L; l++)
        if ((int64_t)h->lev[l].A.n * h->lev[l].A.n * K <= kOpWorkM) return l;
    return L;
}

// Blocks of a grid-stride kernel: one thread per item up to two waves, else
// one wave of what stays resident (a grid that is no multiple of it leaves SMs
// with blocks to spare at the end).
template <typename F>
int wave_grid(const MultiWS &W, F *kernel, int64_t items) {
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kMB, 0) != cudaSuccess || per < 1) per = 1;
    const int64_t want = (items + kMB - 1) / kMB, wave = (int64_t)W.sms * per;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want <= 2 * wave ? want : wave, W.grid));
}

// Threads per block of the coarse levels' kernels (few rows spread over the SMs).
inline int block_of(const MultiWS &W, int64_t items) {
    return items <= (int64_t)W.sms * 64 ? 64 : items <= (int64_t)W.sms * 128 ? 128 : kMB;
}

// Threads up to which a coarse level waits for latency and its rows load 16
// entries per chunk (k_down_c, k_post_c), else 4 at a higher residency: 55,000
// threads (13,800 rows x 8 in float64) 19.4 us with 16 and 22.3 with 4, 110,000
// (x 32 in float32) 26.1 and 11.5, 220,000 (x 32 in float64) 52.9 and 32.4.
constexpr int kChunkThreadsM = 65536;

// Blocks of the level-0 sweeps and of q = A p. In float32 one wave of what
// stays resident; in float64, which its pipe bounds, eight blocks per SM
// whatever stays: 96^3 x 32 down sweep 1,541 us in one wave and 1,435 so, x 8
// 391 and 360, post sweep 391 and 374, q = A p 364 and 345. In float32 eight
// per SM cost 152.2 ms a solve (x 32) for 148.3.
template <typename T, typename F>
int sweep_grid(const MultiWS &W, F *kernel, int64_t items) {
    return sizeof(T) == 8 ? W.grid : wave_grid(W, kernel, items);
}

template <typename T, bool FCG, int K>
int launch_vcycle_m(amg_hier *h, MultiWS &W, cudaStream_t s) {
    using P = MP<T>;
    constexpr int V = VW<T>::V;
    auto &lev = h->lev;
    const int L = direct_level_m(h, K);  // levels 0..L-1 are swept
    const bool pdl = h->pdl;
    CtlM *ctl = W.ctl;
    Level &l0 = lev[0];
    MultiLevel &m0 = W.lev[0];
    const int64_t items0 = (int64_t)l0.A.n * (K / V);
    const T *b0;
    if constexpr (sizeof(T) == 4) b0 = W.r32;
    else b0 = W.r;
    if (L == 0) {
        // single level: z = A^{-1} r through the coarse kernel (float32 rounding as the V-cycle's)
        set_error("pcg_solve_multi: single-level hierarchy not supported by the multi-column path");
        return AMG_ERR_ARG;
    }
    const bool gs = h->gs_nu > 0;
    if (gs) launch_gs_m<T, K>(h, W, 0, true, b0, P::xpre(m0), s);
    WITH_COLS_M(l0.S, (launch_k(pdl, k_down_m<T, IDX, K, kUnroll, true>,
                                sweep_grid<T>(W, k_down_m<T, IDX, K, kUnroll, true>, items0), kMB, s, l0.A.n, l0.S.sptr,
                                cols, P::val(l0), P::xpre(m0), b0, P::p(l0), P::t(m0), ctl)));
    for (int l = 0; l < L; l++) {
        Level &lv = lev[l];
        MultiLevel &mv = W.lev[l];
        const int n = lv.A.n;
        const int64_t items = (int64_t)n * (K / V), citems = (int64_t)lv.nc * (K / V);
        if (l > 0) {
            if (gs) launch_gs_m<T, K>(h, W, l, true, P::b(mv), P::xpre(mv), s);
            const int blk = block_of(W, items), g = (int)((items + blk - 1) / blk);
            if (items <= kChunkThreadsM)
                WITH_COLS_M(lv.S, (launch_k(pdl, k_down_c<T, IDX, K, kUnrollSmall>, g, blk, s, n, lv.S.sptr, cols,
                                            P::val(lv), pats, P::xpre(mv), P::b(mv), P::p(lv), P::t(mv), ctl)));
            else
                WITH_COLS_M(lv.S, (launch_k(pdl, k_down_m<T, IDX, K, kUnroll, false>, grid_of(items), kMB, s, n,
                                            lv.S.sptr, cols, P::val(lv), P::xpre(mv), P::b(mv), P::p(lv), P::t(mv),
                                            ctl)));
        }
        const int cblk = block_of(W, citems), cg = (int)((citems + cblk - 1) / cblk);
        if (l + 1 == L)
            launch_k(pdl, k_restrict_m<T, double, false, K>, cg, cblk, s, lv.nc, lv.rptr, lv.ridx, P::t(mv), W.bL,
                     nullptr, nullptr, ctl);
        else
            launch_k(pdl, k_restrict_m<T, T, true, K>, cg, cblk, s, lv.nc, lv.rptr, lv.ridx, P::t(mv),
                     P::b(W.lev[l + 1]), P::dinv(lev[l + 1]), P::xpre(W.lev[l + 1]), ctl);
    }
    if (h->coarse_iter)
        PCG_TRY(launch_coarse_iter<T>(h, W.cws, W.bL, P::x(W.lev[L]), &ctl->done, ctl->active, s));
    else
        launch_k(pdl, k_coarse_m<T, K>, grid_of((int64_t)lev[L].A.n * (K / 2) * 32), kMB, s, lev[L].A.n,
                 h->op_first && h->op[L] ? h->op[L] : h->Ainv, W.bL, P::x(W.lev[L]), ctl);
    for (int l = L - 1; l >= 1; l--) {
        Level &lv = lev[l];
        MultiLevel &mv = W.lev[l];
        const int n = lv.A.n;
        const int64_t items = (int64_t)n * (K / V);
        const int blk = block_of(W, items), g = (int)((items + blk - 1) / blk);
        launch_k(pdl, k_prolong_m<T, K>, g, blk, s, n, P::xpre(mv), P::p(lv), lv.agg, P::x(W.lev[l + 1]), P::xp(mv),
                 ctl);
        if (gs)
            launch_gs_m<T, K>(h, W, l, false, P::b(mv), P::x(mv), s);
        else if (items <= kChunkThreadsM)
            WITH_COLS_M(lv.S, (launch_k(pdl, k_post_c<T, IDX, K, kUnrollSmall>, g, blk, s, n, lv.S.sptr, cols,
                                        P::val(lv), pats, P::xp(mv), P::b(mv), P::dinv(lv), P::x(mv), ctl)));
        else
            WITH_COLS_M(lv.S, (launch_k(pdl, k_post_m<T, T, false, false, IDX, K, kUnroll, false>, grid_of(items),
                                        kMB, s, n, lv.S.sptr, cols, P::val(lv), P::xp(mv), P::b(mv), P::dinv(lv),
                                        P::x(mv), (const double *)nullptr, (const double *)nullptr,
                                        (double *)nullptr, ctl)));
    }
    launch_k(pdl, k_prolong_m<T, K>, wave_grid(W, k_prolong_m<T, K>, items0), kMB, s, l0.A.n, P::xpre(m0), P::p(l0),
             l0.agg, P::x(W.lev[1]), P::xp(m0), ctl);
    if (gs) {
        launch_gs_m<T, K>(h, W, 0, false, b0, P::x(m0), s);
        launch_k(pdl, k_gs_finish0_m<T, FCG, K>, wave_grid(W, k_gs_finish0_m<T, FCG, K>, items0), kMB, s, l0.A.n,
                 (const T *)P::x(m0), W.r, W.q, W.z, W.partials, ctl);
        PCG_LAUNCH_CK();
        return AMG_OK;
    }
    WITH_COLS_M(l0.S, (launch_k(pdl, k_post_m<T, double, true, FCG, IDX, K, kUnroll, true>,
                                sweep_grid<T>(W, k_post_m<T, double, true, FCG, IDX, K, kUnroll, true>, items0), kMB, s,
                                l0.A.n, l0.S.sptr, cols, P::val(l0), P::xp(m0), b0, P::dinv(l0), W.z, W.r, W.q,
                                W.partials, ctl)));
    PCG_LAUNCH_CK();
    return AMG_OK;
}

// k_residual_m of `mode` (INIT: the pending columns' first residual).
template <bool INIT, int K>
void launch_residual_m(amg_hier *h, MultiWS &W, int mode, cudaStream_t s) {
    Level &l0 = h->lev[0];
    MultiLevel &m0 = W.lev[0];
    const int n = l0.A.n;
    const int64_t items = (int64_t)n * (K / 2);
#define PCG_RESIDUAL_M(MODE)                                                                                         \
    WITH_COLS_M(l0.S, (launch_k(h->pdl, k_residual_m<INIT, MODE, IDX, K>,                                           \
                                wave_grid(W, k_residual_m<INIT, MODE, IDX, K>, items), kMB, s, n, l0.S.sptr, cols,  \
                                l0.S.v64, W.b, W.x, W.r, W.r32, l0.dinv32, m0.xpre32, l0.dinv, m0.xpre64,           \
                                W.partials, W.ctl, W.hist, W.hist_cap)))
    if (mode == AMG_MODE_FCG32) PCG_RESIDUAL_M(AMG_MODE_FCG32);
    else PCG_RESIDUAL_M(AMG_MODE_PCG64);
#undef PCG_RESIDUAL_M
}

template <int K>
int launch_iteration_m(amg_hier *h, MultiWS &W, int mode, cudaStream_t s) {
    Level &l0 = h->lev[0];
    MultiLevel &m0 = W.lev[0];
    const int n = l0.A.n;
    const int64_t items = (int64_t)n * (K / 2);
    if (mode == AMG_MODE_FCG32) PCG_TRY((launch_vcycle_m<float, true, K>(h, W, s)));
    else if (h->coarse_iter) PCG_TRY((launch_vcycle_m<double, true, K>(h, W, s)));  // flexible: FCG(1) beta
    else PCG_TRY((launch_vcycle_m<double, false, K>(h, W, s)));
    launch_k(h->pdl, k_axpy_m<K>, wave_grid(W, k_axpy_m<K>, items), kMB, s, n, W.z, W.p, W.ctl);
    WITH_COLS_M(l0.S, (launch_k(h->pdl, k_spmm_m<IDX, K>, sweep_grid<double>(W, k_spmm_m<IDX, K>, items), kMB, s, n, l0.S.sptr,
                                cols, l0.S.v64, W.p, W.q, W.partials, W.ctl)));
    // half a wave of the update: its partials are what its last block reads
    if (mode == AMG_MODE_FCG32)
        launch_k(h->pdl, k_update_m<AMG_MODE_FCG32, K>, (wave_grid(W, k_update_m<AMG_MODE_FCG32, K>, items) + 1) / 2,
                 kMB, s, n, W.p, W.q, W.x, W.r, W.r32, l0.dinv32, m0.xpre32, l0.dinv, m0.xpre64, W.partials, W.ctl,
                 W.hist, W.hist_cap);
    else
        launch_k(h->pdl, k_update_m<AMG_MODE_PCG64, K>, (wave_grid(W, k_update_m<AMG_MODE_PCG64, K>, items) + 1) / 2,
                 kMB, s, n, W.p, W.q, W.x, W.r, W.r32, l0.dinv32, m0.xpre32, l0.dinv, m0.xpre64, W.partials, W.ctl,
                 W.hist, W.hist_cap);
    launch_residual_m<false, K>(h, W, mode, s);
    PCG_LAUNCH_CK();
    return AMG_OK;
}

// First residual, ||b|| and state of the pending columns only.
template <int K>
int launch_init_residual_m(amg_hier *h, MultiWS &W, int mode, cudaStream_t s) {
    launch_residual_m<true, K>(h, W, mode, s);
    PCG_LAUNCH_CK();
    return AMG_OK;
}

template <int K>
int launch_prefix_m(amg_hier *h, MultiWS &W, int mode, cudaStream_t s) {
    int64_t nk = (int64_t)h->lev[0].A.n * K;
    k_zero_m<<<grid_of(nk), kMB, 0, s>>>(W.p, nk);
    k_zero_m<<<grid_of(nk), kMB, 0, s>>>(W.q, nk);
    PCG_LAUNCH_CK();
    return launch_init_residual_m<K>(h, W, mode, s);
}

// Whole multi-column solve as one graph (prefix, then a device-side while
// loop of two iterations per body), as in the single-column path.
template <int K>
int build_graph_m(amg_hier *h, MultiWS &W, int mode) {
    if (!h->cap_stream) PCG_CK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    cudaStream_t cs = h->cap_stream;
    PCG_CK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    int st = launch_prefix_m<K>(h, W, mode, cs);
    cudaGraph_t g = nullptr;
    cudaGraphConditionalHandle hc = 0;
    cudaStreamCaptureStatus cst;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    cudaGraphNodeParams cp = {};
    cudaGraphNode_t cnode = nullptr;
    cudaError_t e = cudaSuccess;
    if (!st) e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, &g, nullptr, nullptr, nullptr);
    if (!st && e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&hc, g, 1, cudaGraphCondAssignDefault);
    if (!st && e == cudaSuccess) {
        k_set_cond_m<<<1, 32, 0, cs>>>(hc, W.ctl, 0);
        e = cudaGetLastError();
    }
    if (!st && e == cudaSuccess) e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, &g, &deps, nullptr, &nd);
    if (!st && e == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = hc;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        e = cudaGraphAddNode(&cnode, g, deps, nullptr, nd, &cp);
    }
    if (!st && e == cudaSuccess)
        e = cudaStreamUpdateCaptureDependencies(cs, &cnode, nullptr, 1, cudaStreamSetCaptureDependencies);
    cudaGraph_t full = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(cs, &full);
    if (st || e != cudaSuccess || e2 != cudaSuccess) {
        if (full) cudaGraphDestroy(full);
        if (!st) st = cuda_fail(e != cudaSuccess ? e : e2, "multi solve graph capture", __FILE__, __LINE__);
        return st;
    }
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        st = launch_iteration_m<K>(h, W, mode, cs);
        if (!st) st = launch_iteration_m<K>(h, W, mode, cs);
        if (!st) k_set_cond_m<<<1, 32, 0, cs>>>(hc, W.ctl, 1);
        cudaGraph_t bout = body;
        e = cudaStreamEndCapture(cs, &bout);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (st || e != cudaSuccess) {
        cudaGraphDestroy(full);
        if (!st) st = cuda_fail(e, "multi solve graph body capture", __FILE__, __LINE__);
        return st;
    }
    e = cudaGraphInstantiate(&W.gexec[mode], full, 0);
    cudaGraphDestroy(full);
    if (e != cudaSuccess) {
        W.gexec[mode] = nullptr;
        return cuda_fail(e, "cudaGraphInstantiate (multi)", __FILE__, __LINE__);
    }
    return AMG_OK;
}

bool is_dev(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Workspace of K columns (reallocated when K or the history length grows).
int ensure_ws(amg_hier *h, int K, int maxit) {
    MultiWS &W = h->multi;
    if (W.K == K && W.hist_cap >= maxit + 1) return AMG_OK;
    mws_free(h->mem, W);
    return mws_alloc(h, h->mem, W, K, maxit + 1 > 1001 ? maxit + 1 : 1001, 3);
}

template <int K>
int solve_multi_k(amg_hier *h, int k, const double *B, double *X, double rtol, int maxit, int *iters,
                  double *res_hist, cudaStream_t s) {
    PCG_TRY(ensure_ws(h, K, maxit));
    MultiWS &W = h->multi;
    int n = h->lev[0].A.n;
    int64_t nk = (int64_t)n * K;
    int64_t nkk = (int64_t)n * k;
    Mem &M = h->mem;
    M.stream = s;
    // inputs into the internal n x K block (through a device staging copy when on the host)
    const double *bsrc = B, *xsrc = X;
    double *stage = nullptr;
    bool bdev = is_dev(B), xdev = is_dev(X);
    if (!bdev || !xdev) PCG_TRY(alloc(M, &stage, (size_t)nkk));
    if (!bdev) {
        PCG_CK(cudaMemcpyAsync(stage, B, sizeof(double) * nkk, cudaMemcpyHostToDevice, s));
        bsrc = stage;
    }
    k_pack<<<grid_of(nk), kMB, 0, s>>>(bsrc, k, W.b, K, n);
    if (!xdev) {
        PCG_CK(cudaMemcpyAsync(stage, X, sizeof(double) * nkk, cudaMemcpyHostToDevice, s));
        xsrc = stage;
    }
    k_pack<<<grid_of(nk), kMB, 0, s>>>(xsrc, k, W.x, K, n);
    PCG_LAUNCH_CK();
    CtlM c0;
    memset(&c0, 0, sizeof(c0));
    c0.rtol = rtol;
    c0.maxit = maxit;
    c0.mode = h->mode;
    c0.flex = h->coarse_iter;
    c0.k = k;
    c0.K = K;
    for (int q = 0; q < K; q++) c0.pending[q] = 1;
    *W.ctl_host = c0;
    PCG_CK(cudaMemcpyAsync(W.ctl, W.ctl_host, sizeof(CtlM), cudaMemcpyHostToDevice, s));
    int mode = h->mode;
    bool graph = h->use_graph;
    if (graph && !W.gexec[mode]) {
        if (build_graph_m<K>(h, W, mode) != AMG_OK) graph = false;
    }
    if (graph) {
        PCG_CK(cudaGraphLaunch(W.gexec[mode], s));
        PCG_CK(cudaMemcpyAsync(W.ctl_host, W.ctl, sizeof(CtlM), cudaMemcpyDeviceToHost, s));
        PCG_CK(cudaStreamSynchronize(s));
    } else {
        PCG_TRY(launch_prefix_m<K>(h, W, mode, s));
        int launched = 0;
        for (;;) {
            PCG_CK(cudaMemcpyAsync(W.ctl_host, W.ctl, sizeof(CtlM), cudaMemcpyDeviceToHost, s));
            PCG_CK(cudaStreamSynchronize(s));
            if (W.ctl_host->done || launched >= maxit) break;
            for (int q = 0; q < 4 && launched < maxit; q++, launched++) PCG_TRY(launch_iteration_m<K>(h, W, mode, s));
        }
    }
    CtlM &c = *W.ctl_host;
    double *xdst = xdev ? X : stage;
    k_unpack<<<grid_of(nkk), kMB, 0, s>>>(W.x, K, xdst, k, n, W.ctl);
    PCG_LAUNCH_CK();
    if (!xdev) PCG_CK(cudaMemcpyAsync(X, stage, sizeof(double) * nkk, cudaMemcpyDeviceToHost, s));
    if (res_hist) {
        int hl = maxit + 1;
        for (int q = 0; q < k; q++)
            PCG_CK(cudaMemcpyAsync(res_hist + (int64_t)q * hl, W.hist + (int64_t)q * W.hist_cap,
                                   sizeof(double) * (c.iter[q] + 1), cudaMemcpyDefault, s));
    }
    PCG_CK(cudaStreamSynchronize(s));
    if (stage) release(M, stage);
    int st = AMG_OK;
    for (int q = 0; q < k; q++) {
        if (iters) iters[q] = c.iter[q];
        h->multi_status[q] = c.status[q];
        h->multi_true_rel[q] = c.true_rel[q];
        if (c.status[q] != AMG_OK && st == AMG_OK) st = c.status[q];
    }
    h->multi_k = k;
    if (st) set_error("pcg_solve_multi: some columns failed (status %d; see amg_multi_info)", st);
    return st;
}

}  // namespace

// Whether the multi-column kernels can smooth h by Gauss-Seidel: every level
// with sweeps has blocks whose size divides 32 and at most kGsPartM
// already-updated in-block entries per row in each pass (one-warp sweeps).
bool gs_multi_ok(const amg_hier *h) {
    if (h->gs_nu <= 0) return true;
    for (size_t l = 0; l + 1 < h->lev.size(); l++) {
        const Level &lv = h->lev[l];
        int nb = gs_rows(lv.A.n, h->gs_blocks);
        if (nb > 32 || 32 % nb) return false;
        for (int d = 0; d < 2; d++)
            if (lv.gs_w[d] < 0 || lv.gs_w[d] > kGsPartM) return false;
    }
    return true;
}

// Allocates a K-column workspace; which: 1 float32 V-cycle vectors,
// 2 float64 V-cycle vectors, 3 both.
int mws_alloc(amg_hier *h, Mem &M, MultiWS &W, int K, int hist_cap, int which) {
    int L = (int)h->lev.size() - 1;
    int n0 = h->lev[0].A.n;
    int64_t nk = (int64_t)n0 * K;
    W.K = K;
    W.hist_cap = hist_cap;
    PCG_TRY(alloc(M, &W.b, nk));
    PCG_TRY(alloc(M, &W.x, nk));
    PCG_TRY(alloc(M, &W.r, nk));
    PCG_TRY(alloc(M, &W.z, nk));
    PCG_TRY(alloc(M, &W.p, nk));
    PCG_TRY(alloc(M, &W.q, nk));
    PCG_TRY(alloc(M, &W.r32, nk));
    W.lev.assign(L + 1, MultiLevel{});
    for (int l = 0; l <= L; l++) {
        int64_t m = (int64_t)h->lev[l].A.n * K;
        MultiLevel &v = W.lev[l];
        if (which & 1) {
            PCG_TRY(alloc(M, &v.b32, m));
            PCG_TRY(alloc(M, &v.x32, m));
            PCG_TRY(alloc(M, &v.t32, m));
            PCG_TRY(alloc(M, &v.xpre32, m));
            PCG_TRY(alloc(M, &v.xp32, m));
        }
        if (which & 2) {
            PCG_TRY(alloc(M, &v.b64, m));
            PCG_TRY(alloc(M, &v.x64, m));
            PCG_TRY(alloc(M, &v.t64, m));
            PCG_TRY(alloc(M, &v.xpre64, m));
            PCG_TRY(alloc(M, &v.xp64, m));
        }
    }
    PCG_TRY(alloc(M, &W.bL, (int64_t)h->lev[direct_level_m(h, K)].A.n * K));
    W.flex = h->coarse_iter;
    if (h->coarse_iter) PCG_TRY(cws_alloc(h, M, W.cws, K));
    int sms = 0;
    PCG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    W.sms = sms;
    int64_t want = (nk + kMB - 1) / kMB;
    int64_t cap = (int64_t)sms * 8;
    W.grid = (int)(want < cap ? want : cap);
    if (W.grid < 1) W.grid = 1;
    PCG_TRY(alloc(M, &W.partials, (size_t)2 * K * W.grid));
    PCG_TRY(alloc(M, &W.ctl, 1));
    PCG_TRY(alloc(M, &W.hist, (size_t)K * W.hist_cap));
    if (M.dry) return AMG_OK;
    PCG_CK(cudaMemsetAsync(W.ctl, 0, sizeof(CtlM), M.stream));
    PCG_CK(cudaMallocHost(&W.ctl_host, sizeof(CtlM)));
    return AMG_OK;
}

// Device bytes that mws_alloc takes for this workspace shape (exact: the
// same requests, counted by a dry-run pool).
size_t mws_bytes(amg_hier *h, int K, int hist_cap, int which) {
    Mem M;
    M.dry = true;
    MultiWS W;
    if (mws_alloc(h, M, W, K, hist_cap, which)) return (size_t)-1;
    return M.bytes;
}

void mws_free(Mem &M, MultiWS &W) {
    for (auto &g : W.gexec) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    if (W.step_exec) cudaGraphExecDestroy(W.step_exec);
    if (W.step_graph) cudaGraphDestroy(W.step_graph);
    W.step_exec = nullptr;
    W.step_graph = nullptr;
    W.step_iters = 0;
    W.step_mode = -1;
    release(M, W.b);
    release(M, W.x);
    release(M, W.r);
    release(M, W.z);
    release(M, W.p);
    release(M, W.q);
    release(M, W.r32);
    for (auto &v : W.lev) {
        release(M, v.b32); release(M, v.x32); release(M, v.t32); release(M, v.xpre32); release(M, v.xp32);
        release(M, v.b64); release(M, v.x64); release(M, v.t64); release(M, v.xpre64); release(M, v.xp64);
    }
    W.lev.clear();
    release(M, W.bL);
    cws_free(M, W.cws);
    release(M, W.partials);
    release(M, W.ctl);
    release(M, W.hist);
    if (W.ctl_host) cudaFreeHost(W.ctl_host);
    W.ctl_host = nullptr;
    W.K = 0;
    W.hist_cap = 0;
}

void free_multi(amg_hier *h) { mws_free(h->mem, h->multi); }

namespace {

// Column c of a new request: b and x0 in, and p = q = 0 (the first
// iteration's p = z + 0 p and FCG's z.q_old must not see an earlier
// occupant's values).
__global__ void k_col_put(const double *__restrict__ b, const double *__restrict__ x0, double *__restrict__ B,
                          double *__restrict__ X, double *__restrict__ P, double *__restrict__ Q, int K, int c,
                          int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t e = (int64_t)i * K + c;
    B[e] = b[i];
    X[e] = x0[i];
    P[e] = 0.0;
    Q[e] = 0.0;
}

// Marks new columns for initialisation and wakes the solve up.
__global__ void k_admit(CtlM *ctl, unsigned mask) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    for (int c = 0; c < ctl->K; c++)
        if (mask & (1u << c)) {
            ctl->pending[c] = 1;
            ctl->active[c] = 0;
            ctl->status[c] = AMG_OK;
        }
    ctl->done = 0;
}

// Only the new columns' p and q were cleared (by their put): the running
// columns keep their search directions.
template <int K>
int mws_init_pending(amg_hier *h, MultiWS &W, int mode, cudaStream_t s) {
    return launch_init_residual_m<K>(h, W, mode, s);
}

}  // namespace

// Resets a workspace's state: no column in use, solve idle.
int mws_reset(MultiWS &W, int mode, double rtol, int maxit, cudaStream_t s) {
    CtlM c0;
    memset(&c0, 0, sizeof(c0));
    c0.rtol = rtol;
    c0.maxit = maxit;
    c0.mode = mode;
    c0.flex = W.flex;
    c0.k = W.K;
    c0.K = W.K;
    c0.done = 1;
    *W.ctl_host = c0;
    PCG_CK(cudaMemcpyAsync(W.ctl, W.ctl_host, sizeof(CtlM), cudaMemcpyHostToDevice, s));
    PCG_CK(cudaStreamSynchronize(s));
    return AMG_OK;
}

int mws_put_column(MultiWS &W, int c, const double *b_dev, const double *x_dev, int n, cudaStream_t s) {
    k_col_put<<<(n + kMB - 1) / kMB, kMB, 0, s>>>(b_dev, x_dev, W.b, W.x, W.p, W.q, W.K, c, n);
    PCG_LAUNCH_CK();
    return AMG_OK;
}

// Starts the columns in mask: residual, ||b|| and state of each, while the
// other columns keep their place in their own iterations.
int mws_admit(amg_hier *h, MultiWS &W, int mode, unsigned mask, cudaStream_t s) {
    k_admit<<<1, 32, 0, s>>>(W.ctl, mask);
    PCG_LAUNCH_CK();
    switch (W.K) {
        case 4: return mws_init_pending<4>(h, W, mode, s);
        case 8: return mws_init_pending<8>(h, W, mode, s);
        case 16: return mws_init_pending<16>(h, W, mode, s);
        default: return mws_init_pending<32>(h, W, mode, s);
    }
}

// `iterations` iterations of every active column (kernels of finished
// columns do no work), then the state is copied to the pinned host mirror.
// The chunk is captured once as a graph (kept in W) that every later call
// replays; launch = 0 only captures it.
int mws_iterate(amg_hier *h, MultiWS &W, int mode, int iterations, cudaStream_t s, int launch) {
    if (!W.step_exec || W.step_iters != iterations || W.step_mode != mode) {
        if (W.step_exec) cudaGraphExecDestroy(W.step_exec);
        if (W.step_graph) cudaGraphDestroy(W.step_graph);
        W.step_exec = nullptr;
        W.step_graph = nullptr;
        if (!h->cap_stream) PCG_CK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
        cudaStream_t cs = h->cap_stream;
        PCG_CK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        int st = AMG_OK;
        for (int k = 0; k < iterations && !st; k++) {
            switch (W.K) {
                case 4: st = launch_iteration_m<4>(h, W, mode, cs); break;
                case 8: st = launch_iteration_m<8>(h, W, mode, cs); break;
                case 16: st = launch_iteration_m<16>(h, W, mode, cs); break;
                default: st = launch_iteration_m<32>(h, W, mode, cs); break;
            }
        }
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(cs, &g);
        if (st) {
            if (g) cudaGraphDestroy(g);
            return st;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&W.step_exec, g, 0);
        if (e != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            W.step_exec = nullptr;
            return cuda_fail(e, "serving step graph", __FILE__, __LINE__);
        }
        W.step_graph = g;
        W.step_iters = iterations;
        W.step_mode = mode;
    }
    if (!launch) return AMG_OK;
    PCG_CK(cudaGraphLaunch(W.step_exec, s));
    PCG_CK(cudaMemcpyAsync(W.ctl_host, W.ctl, sizeof(CtlM), cudaMemcpyDeviceToHost, s));
    return AMG_OK;
}

int solve_multi_impl(amg_hier *h, int k, const double *B, double *X, double rtol, int maxit, int *iters,
                     double *res_hist, cudaStream_t s) {
    if (k < 1 || k > kMaxK || !B || !X || !(rtol >= 0.0) || maxit < 0) {
        set_error("pcg_solve_multi: bad arguments (1 <= k <= 32, rtol >= 0, maxit >= 0)");
        return AMG_ERR_ARG;
    }
    if (h->lev.size() < 2) {
        set_error("pcg_solve_multi: the hierarchy has a single level; use pcg_solve per column");
        return AMG_ERR_ARG;
    }
    int K = 4;
    while (K < k) K <<= 1;
    switch (K) {
        case 4: return solve_multi_k<4>(h, k, B, X, rtol, maxit, iters, res_hist, s);
        case 8: return solve_multi_k<8>(h, k, B, X, rtol, maxit, iters, res_hist, s);
        case 16: return solve_multi_k<16>(h, k, B, X, rtol, maxit, iters, res_hist, s);
        default: return solve_multi_k<32>(h, k, B, X, rtol, maxit, iters, res_hist, s);
    }
}

}  // namespace pcgamg

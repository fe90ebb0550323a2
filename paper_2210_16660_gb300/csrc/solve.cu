// Solve phase: PCG / FCG(1) preconditioned by one V-cycle per iteration
// (arxiv 2210.16660, Sec. 3.1 Eq. (multiplicative composition) with nu = 1
// and M = D_l1; Sec. 5 flexible CG with a relative-residual stop).
//
// Every sweep streams a sliced-ELL matrix (one warp per 32-row slice,
// coalesced value/column loads, 4 entries of a row loaded ahead of their
// gathers) and fuses the vector work around it.
//
// GB300 note: float64 FMA throughput (~1.25 TFLOP/s) is about what one FMA per
// stored entry needs at full HBM bandwidth, so every float64 sweep does
// exactly one float64 operation per stored entry; anything else is formed
// once per row (D^-1 b, D^-1 b + P x_c, p = z + beta p). The float32 V-cycle
// reads a float32 copy of r (and of D^-1 r) so no conversion happens per entry.
//
// V-cycle (T = float for FCG(1), double for PCG; one structure for both):
//   down   : t = p .* (b - A xpre), xpre = D^-1 b formed by the producer of b
//   restr  : b_{l+1}[I] = sum_{i in G_I} t_i (members in index order), and
//            xpre_{l+1} = D^-1 b_{l+1}
//   coarse : x_L = A_L^{-1} b_L (float64 dense inverse)
//   prolong: xp = xpre + P x_{l+1}
//   post   : z = xp + D^-1 (b - A xp)
// so every sweep gathers one vector per stored entry.
// Krylov (float64): p = z + beta p; q = A p, p.q; x += alpha p,
// r -= alpha q, ||r||^2 (+ r32 or xpre_0); true residual when rtol is met.
//
// Reductions are two-stage and deterministic: each block of the producing
// kernel writes a partial, and every block of the kernel that needs the sum
// adds all partials before its own work (one block also records the scalars
// in struct Ctl). So a reduction costs its consumer one L2 round trip and a
// block sum, and the producer no fence, ticket or serial last block. Sums over
// threads run on the integer pipe (reduce.cuh), and one thread per block forms
// the scalars: a float64 quotient or root costs a warp 560 to 600 clocks.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "reduce.cuh"
#include "sell_row.cuh"

namespace pcgamg {

namespace {

constexpr int kVecBlock = 512;  // largest block of the vector kernels (k_axpy_p, k_update)

template <typename T>
__device__ __forceinline__ T ldg(const T *p) { return __ldg(p); }

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// As write_partials, and true in every thread of the last block to finish,
// after which all partials are complete: for the true residual, whose outcome
// decides whether the loop goes on.
template <int NV>
__device__ __forceinline__ bool publish_partials(double (&a)[NV], double *partials, unsigned *counter) {
    __shared__ bool last;
    write_partials<NV>(a, partials);
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned t = atomicAdd(counter, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    return last;
}

// Reads of the solve's state go to L2. A kernel launched with programmatic
// dependence starts, and drops its SM's L1 lines, while its predecessor still
// runs: a block of the predecessor on that SM may then bring a line of Ctl
// into L1 before another block changes it, and nothing shows that a plain
// load after the wait cannot still hit that line.
template <typename T>
__device__ __forceinline__ T state(const T *p) { return __ldcg(p); }
__device__ __forceinline__ int halted(const Ctl *c) { return state(&c->halt); }
// The same by one thread for the block, for kernels of many blocks: L2 serves the
// warps' requests for the one sector one after another (k_restrict and k_prolong
// of 128^3: 21.68 -> 21.43 ms a mixed solve, 31.17 -> 30.92 float64). Every
// thread of the block calls it.
__device__ __forceinline__ int halted_block(const Ctl *c) {
    return __syncthreads_or(threadIdx.x == 0 ? halted(c) : 0);
}

// Ctl::halt: whether the iteration's kernels run
constexpr int kRun = 0, kCheck = 1, kEnded = 2;

__device__ __forceinline__ void finish(Ctl *c) {
    c->done = 1;
    c->halt = kEnded;
    c->status = AMG_OK;
}

__device__ __forceinline__ void fail(Ctl *c, int status) {
    c->done = 2;
    c->halt = kEnded;
    c->status = status;
}

// Outcome of the iteration whose update left g partial sums of ||r||^2:
// kRun, or why the kernels that follow must not run (kCheck: rtol met, the
// true residual is formed next; kEnded). Called by every thread of every block
// of one kernel; one thread records the outcome in ctl->halt. A block that
// starts after that finds it there, and takes the same way as on its own: the
// flag is read by one thread for the whole block, as another block may be
// writing it.
__device__ __forceinline__ int step_outcome(const double *pc, int g, Ctl *ctl, double *hist) {
    __shared__ int out;
    __shared__ double srr;
    int halt = kRun, it = 0, maxit = 0;
    double stop2 = 0.0;
    if (threadIdx.x == 0) {
        halt = halted(ctl);
        it = state(&ctl->iter);
        maxit = state(&ctl->maxit);
        stop2 = state(&ctl->stop2);
    }
    double rr[1];
    sum_partials<1>(pc, g, rr);
    if (threadIdx.x == 0) {
        int o = halt;
        if (o == kRun) {
            o = !isfinite(rr[0]) ? kEnded : rr[0] <= stop2 ? kCheck : it >= maxit ? kEnded : kRun;
            if (blockIdx.x == 0) {
                if (o == kCheck) ctl->halt = kCheck;
                else if (o == kEnded) fail(ctl, isfinite(rr[0]) ? AMG_ERR_NOCONV : AMG_ERR_NAN);
            }
        }
        out = o;
        srr = halt == kRun ? rr[0] : -1.0;
    }
    __syncthreads();
    // the history's root and quotient in a thread that nothing waits for
    if (blockIdx.x == 0 && threadIdx.x == 32 && !(srr < 0.0)) {
        const double rel = sqrt(srr) / state(&ctl->bnorm);
        ctl->rel = rel;
        hist[state(&ctl->iter)] = rel;
    }
    return out;
}

#define SELL_ROW_BEGIN                                               \
    int s_ = i >> 5, lane_ = i & 31;                                 \
    int32_t base_ = ldg(sptr + s_);                                  \
    int w_ = (ldg(sptr + s_ + 1) - base_) >> 5;                      \
    const IDX *c_ = col + base_ + lane_;                             \
    const auto *a_ = val + base_ + lane_;

// ------------------------------------------------------------ V-cycle sweeps
template <typename T>
struct Occ { static constexpr int kMinBlocks = sizeof(T) == 4 ? 6 : 4; };
// Sweeps with 16-entry chunks hold two chunks (the current one and the one
// in flight) in registers: two float32 blocks per SM, one float64.
template <typename T, int U>
struct SweepOcc {
    static constexpr int kMinBlocks = U <= 4 ? Occ<T>::kMinBlocks
                                      : U == kWholeRow ? 1
                                      : U == kPatRow ? (sizeof(T) == 4 ? 3 : 1)
                                                     : (sizeof(T) == 4 ? 2 : 1);
};

// The V-cycle sweeps, restriction and prolongation read their first row's
// static data (matrix entries, weights, aggregate maps: written only by
// setup and refresh) before pdl_enter(), so it arrives while the preceding
// kernel drains; what a preceding kernel wrote is read through after_wait()
// pointers once the wait has returned.

// Pre-smooth from zero, residual, weighted restriction input:
// t_i = p_i (b_i - sum_j a_ij xpre_j), xpre = D^-1 b.
// STEP: the first kernel of an iteration that follows another one in the same
// loop body; it reads that iteration's outcome (step_outcome).
template <typename T, typename IDX, int U, bool STREAM, bool STEP>
__global__ void __launch_bounds__(kBlock, SweepOcc<T, U>::kMinBlocks) k_down(
    int n, const int32_t *__restrict__ sptr, const IDX *__restrict__ col, const T *__restrict__ val,
    const IDX *__restrict__ upat, const T *__restrict__ xpre, const T *__restrict__ b,
    const T *__restrict__ p, T *__restrict__ t, const double *pc, int gc, Ctl *ctl, double *hist) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    RowOf<U, STREAM, IDX, T> R;
    T pi = 0;
    if (i < n) {
        R.load(sptr, col, val, i, upat);
        pi = ldg(p + i);
    }
    pdl_enter();
    xpre = after_wait(xpre);
    b = after_wait(b);
    ctl = after_wait(ctl);
    // a kernel that takes an outcome may write the flag: it is read there
    const int halt = STEP ? 0 : halted(ctl);
    if (U != kWholeRow && halt) return;
    if (STEP && step_outcome(after_wait(pc), gc, ctl, hist) != kRun) return;
    for (; i < n; i += stride) {
        const T bi = ldg(b + i);
        T acc = R.dot(i, [&](int j) { return ldg(xpre + j); });
        if (U == kWholeRow && halt) return;
        t[i] = pi * (bi - acc);
        if (i + stride < n) {
            R.load(sptr, col, val, i + stride, upat);
            pi = ldg(p + i + stride);
        }
    }
}

// Down sweep and the restriction it feeds in one launch: thread <-> position of
// the member order (Level::mrow), so the members of a coarse row are slot
// consecutive lanes. t_i = p_i (b_i - sum_j a_ij xpre_j) as in k_down, then
// the slot's lanes are added in member order by shuffles to b_c and
// (dinvc given) xpre_c = dinv_c b_c; t is never stored. Rows left out of the
// coarse space take xp = xpre, for the prolongation by the coarser level's
// kernel (Up). Same values as k_down followed by k_restrict.
template <typename T, typename TO, typename IDX>
struct DownR {
    const int32_t *mrow;
    int npos, nmain, lg;  // positions, positions of members, log2 of the slot
    const int32_t *sptr;
    const IDX *col;
    const T *val;
    const IDX *upat;
    const T *xpre, *b, *p;
    TO *bc;
    const T *dinvc;
    T *xprec, *xp;
    const double *pc;
    int gc;
    Ctl *ctl;
    double *hist;
};

template <typename T, typename TO, typename IDX, int U, bool STREAM, bool STEP>
__global__ void __launch_bounds__(kBlock, SweepOcc<T, U>::kMinBlocks) k_down_r(DownR<T, TO, IDX> a) {
    int pos = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    const int slot = 1 << a.lg;
    RowOf<U, STREAM, IDX, T> R;
    int row = -1, next = -1;
    T pi = 0, dc = 0;
    auto fetch = [&](int q) {  // static data of position q, whose row is `row`
        if (row >= 0 && q < a.nmain) {
            R.load(a.sptr, a.col, a.val, row, a.upat);
            pi = ldg(a.p + row);
            if (a.dinvc && (q & (slot - 1)) == 0) dc = ldg(a.dinvc + (q >> a.lg));
        }
    };
    if (pos < a.npos) {
        row = ldg(a.mrow + pos);
        fetch(pos);
    }
    pdl_enter();
    const T *xpre = after_wait(a.xpre), *b = after_wait(a.b);
    Ctl *ctl = after_wait(a.ctl);
    const int halt = STEP ? 0 : halted(ctl);
    if (U != kWholeRow && halt) return;
    if (STEP && step_outcome(after_wait(a.pc), a.gc, ctl, a.hist) != kRun) return;
    for (; pos < a.npos; pos += stride) {  // npos and nmain are multiples of 32: a warp stays whole
        if (pos + stride < a.npos) next = ldg(a.mrow + pos + stride);
        if (pos >= a.nmain) {
            if (row >= 0) {
                const T x = ldg(xpre + row);
                if (U == kWholeRow && halt) return;
                a.xp[row] = x;
            }
        } else {
            T t = 0;
            if (row >= 0) {
                const T bi = ldg(b + row);
                const T acc = R.dot(row, [&](int j) { return ldg(xpre + j); });
                // rounded product (never contracted into the sum), as k_down stores t
                t = mul_rn(pi, bi - acc);
            }
            T sum = T(0) + t;
            for (int u = 1; u < slot; u++) sum += __shfl_down_sync(0xffffffffu, t, u);
            if (U == kWholeRow && halt) return;
            if (row >= 0 && (pos & (slot - 1)) == 0) {
                const int I = pos >> a.lg;
                a.bc[I] = (TO)sum;
                if (a.dinvc) a.xprec[I] = dc * sum;
            }
        }
        row = next;
        if (pos + stride < a.npos) fetch(pos + stride);
    }
}

// The multi-lane launch shape of the coarse levels: k_down and k_post with
// kMlL lanes per row (MlRow), one row per lane group, the whole of a row's
// first pass (columns and values) loaded before the wait. Same values and
// summation order as k_down / k_post. A warp whose rows lie past the last
// slice leaves before any shuffle; the others keep every lane to the end.
template <typename T, typename IDX>
__global__ void __launch_bounds__(kBlock) k_down_ml(int n, const int32_t *__restrict__ sptr,
                                                    const IDX *__restrict__ col, const T *__restrict__ val,
                                                    const T *__restrict__ xpre, const T *__restrict__ b,
                                                    const T *__restrict__ p, T *__restrict__ t,
                                                    const Ctl *__restrict__ ctl) {
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = gid / kMlL, q = gid % kMlL;
    if ((row >> 5) >= (n + 31) >> 5) return;
    const bool live = row < n;
    MlRow<false, IDX, T> R;
    R.load(sptr, col, val, row, q, live);
    T pi = 0;
    if (live && q == 0) pi = ldg(p + row);
    pdl_enter();
    xpre = after_wait(xpre);
    b = after_wait(b);
    ctl = after_wait(ctl);
    if (halted(ctl)) return;
    T acc = R.dot(row, [&](int j) { return ldg(xpre + j); });
    if (live && q == 0) t[row] = pi * (ldg(b + row) - acc);
}

template <typename T, typename IDX>
__global__ void __launch_bounds__(kBlock) k_post_ml(int n, const int32_t *__restrict__ sptr,
                                                    const IDX *__restrict__ col, const T *__restrict__ val,
                                                    const T *__restrict__ xp, const T *__restrict__ b,
                                                    const T *__restrict__ dinv, T *__restrict__ z,
                                                    const Ctl *__restrict__ ctl) {
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = gid / kMlL, q = gid % kMlL;
    if ((row >> 5) >= (n + 31) >> 5) return;
    const bool live = row < n;
    MlRow<false, IDX, T> R;
    R.load(sptr, col, val, row, q, live);
    T di = 0;
    if (live && q == 0) di = ldg(dinv + row);
    pdl_enter();
    xp = after_wait(xp);
    b = after_wait(b);
    ctl = after_wait(ctl);
    if (halted(ctl)) return;
    T acc = R.dot(row, [&](int j) { return ldg(xp + j); });
    if (live && q == 0) z[row] = ldg(xp + row) + di * (ldg(b + row) - acc);
}

// xp_i = xpre_i + p_i xc[agg_i].
template <typename T>
__global__ void __launch_bounds__(kBlock) k_prolong(int n, const T *__restrict__ xpre, const T *__restrict__ p,
                                                    const int32_t *__restrict__ agg, const T *__restrict__ xc,
                                                    T *__restrict__ xp, const Ctl *__restrict__ ctl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    int a = -1;
    T pw = 0;
    if (i < n) {
        a = ldg(agg + i);
        pw = ldg(p + i);
    }
    pdl_enter();
    xpre = after_wait(xpre);
    xc = after_wait(xc);
    ctl = after_wait(ctl);
    if (halted_block(ctl)) return;
    for (; i < n; i += stride) {
        T x = ldg(xpre + i);
        if (a >= 0) x = fma_rn(pw, ldg(xc + a), x);
        xp[i] = x;
        if (i + stride < n) {
            a = ldg(agg + i + stride);
            pw = ldg(p + i + stride);
        }
    }
}

// Prolongation to the finer level by the kernel that forms x: coarse row I's
// members are mrow[slot I ..] of that level (see Level::mrow), and
// xp_m = xpre_m + p_m x_I for each (the rows left out of the coarse space take
// xp = xpre from that level's down sweep). The first four members and their
// weights are static and loaded before the wait, their xpre with the gathers.
template <typename T>
struct Up {
    const int32_t *mrow;
    int slot;
    const T *p;
    const T *xpre;
    T *xp;
};

template <typename T>
struct UpRow {
    int m[4];
    T p[4], x[4];
    __device__ __forceinline__ void load(const Up<T> &u, int I) {
        const int32_t *src = u.mrow + (int64_t)u.slot * I;
        if (u.slot >= 4) {
            const int4 q = __ldg(reinterpret_cast<const int4 *>(src));
            m[0] = q.x; m[1] = q.y; m[2] = q.z; m[3] = q.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++) m[k] = k < u.slot ? ldg(src + k) : -1;
        }
#pragma unroll
        for (int k = 0; k < 4; k++) p[k] = m[k] >= 0 ? ldg(u.p + m[k]) : T(0);
    }
    __device__ __forceinline__ void gather(const Up<T> &u) {
#pragma unroll
        for (int k = 0; k < 4; k++) x[k] = m[k] >= 0 ? ldg(u.xpre + m[k]) : T(0);
    }
    __device__ __forceinline__ void store(const Up<T> &u, int I, T xc) const {
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (m[k] >= 0) u.xp[m[k]] = fma_rn(p[k], xc, x[k]);
        for (int k = 4; k < u.slot; k++) {
            const int q = ldg(u.mrow + (int64_t)u.slot * I + k);
            if (q >= 0) u.xp[q] = fma_rn(ldg(u.p + q), xc, ldg(u.xpre + q));
        }
    }
};

// Post-smooth z_i = xp_i + dinv_i (b_i - sum_j a_ij xp_j); UP also prolongs
// z to the next finer level. On level 0 (DOT)
// z is written in float64 and the kernel also leaves partial sums of r.z
// (float64 r) and, for FCG(1), z.q_old for k_axpy_p.
template <typename T, typename TZ, bool DOT, bool FCG, typename IDX, int U, bool STREAM, bool UP>
__global__ void __launch_bounds__(kBlock, SweepOcc<T, U>::kMinBlocks) k_post(
    int n, const int32_t *__restrict__ sptr, const IDX *__restrict__ col, const T *__restrict__ val,
    const IDX *__restrict__ upat, const T *__restrict__ xp, const T *__restrict__ b,
    const T *__restrict__ dinv, TZ *__restrict__ z, const double *__restrict__ r64,
    const double *__restrict__ qold, double *partials, const Ctl *ctl, Up<T> up) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    RowOf<U, STREAM, IDX, T> R;
    UpRow<T> ur;
    T di = 0;
    if (i < n) {
        R.load(sptr, col, val, i, upat);
        di = ldg(dinv + i);
        if (UP) ur.load(up, i);
    }
    pdl_enter();
    xp = after_wait(xp);
    b = after_wait(b);
    r64 = after_wait(r64);
    qold = after_wait(qold);
    ctl = after_wait(ctl);
    up.xpre = after_wait(up.xpre);
    // a whole row's gathers do not wait for the flag: it is read beside them
    const int halt = halted(ctl);
    if (U != kWholeRow && halt) return;
    double rz = 0.0, zq = 0.0;
    for (; i < n; i += stride) {
        if (UP) ur.gather(up);
        const T bi = ldg(b + i), xi = ldg(xp + i);
        T acc = R.dot(i, [&](int j) { return ldg(xp + j); });
        if (U == kWholeRow && halt) return;
        TZ zo = (TZ)(xi + di * (bi - acc));
        z[i] = zo;
        if (UP) ur.store(up, i, (T)zo);
        if (DOT) {
            rz += ldg(r64 + i) * (double)zo;
            if (FCG) zq += (double)zo * ldg(qold + i);
        }
        if (i + stride < n) {
            R.load(sptr, col, val, i + stride, upat);
            di = ldg(dinv + i + stride);
            if (UP) ur.load(up, i + stride);
        }
    }
    if (DOT) {
        double sums[FCG ? 2 : 1];
        sums[0] = rz;
        if (FCG) sums[FCG ? 1 : 0] = zq;
        write_partials<FCG ? 2 : 1>(sums, partials);
    }
}

// ------------------------------------------------------------ shared pieces
// b_c[I] = sum of t over the members of aggregate I, in increasing index
// order; PRE also forms xpre_c = dinv_c b_c for the next float64 down sweep.
template <typename T, typename TO, bool PRE>
__global__ void __launch_bounds__(kBlock) k_restrict(int nc, const int32_t *__restrict__ rptr,
                                                     const int32_t *__restrict__ ridx, const T *__restrict__ t,
                                                     TO *__restrict__ bc, const T *__restrict__ dinvc,
                                                     T *__restrict__ xprec, const Ctl *__restrict__ ctl) {
    constexpr int M = 4;  // members read before the wait
    int I = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t k0 = 0, k1 = 0;
    int m[M];
    T dc = 0;
    if (I < nc) {
        k0 = ldg(rptr + I);
        k1 = ldg(rptr + I + 1);
#pragma unroll
        for (int u = 0; u < M; u++) m[u] = k0 + u < k1 ? ldg(ridx + k0 + u) : 0;
        if (PRE) dc = ldg(dinvc + I);
    }
    pdl_enter();
    t = after_wait(t);
    ctl = after_wait(ctl);
    const int halt = threadIdx.x == 0 ? halted(ctl) : 0;  // used before the store, as in halted_block
    T tv[M];
#pragma unroll
    for (int u = 0; u < M; u++) tv[u] = k0 + u < k1 ? ldg(t + m[u]) : T(0);
    T s = 0;
#pragma unroll
    for (int u = 0; u < M; u++)
        if (k0 + u < k1) s += tv[u];
    for (int32_t k = k0 + M; k < k1; k++) s += ldg(t + ldg(ridx + k));
    if (__syncthreads_or(halt) || I >= nc) return;
    bc[I] = (TO)s;
    if (PRE) xprec[I] = dc * s;
}

// Smoothed aggregation: b_c[I] = sum over the rows i of P's column I
// (increasing i) of P_iI res_i, res = b - A xpre left by the down sweep
// (launched with unit weights); PRE also forms xpre_c = dinv_c b_c.
template <typename T, typename TO, bool PRE>
__global__ void __launch_bounds__(kBlock) k_restrict_sa(int nc, const int32_t *__restrict__ trp,
                                                        const int32_t *__restrict__ tri, const T *__restrict__ tv,
                                                        const T *__restrict__ res, TO *__restrict__ bc,
                                                        const T *__restrict__ dinvc, T *__restrict__ xprec,
                                                        const Ctl *__restrict__ ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nc) return;
    T s = 0;
    for (int32_t q = ldg(trp + I); q < ldg(trp + I + 1); q++) s += ldg(tv + q) * ldg(res + ldg(tri + q));
    bc[I] = (TO)s;
    if (PRE) xprec[I] = ldg(dinvc + I) * s;
}

// Smoothed aggregation: xp_i = xpre_i + sum over row i of P of P_iJ xc_J.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_prolong_sa(int n, const int32_t *__restrict__ prp,
                                                       const int32_t *__restrict__ pci, const T *__restrict__ pv,
                                                       const T *__restrict__ xpre, const T *__restrict__ xc,
                                                       T *__restrict__ xp, const Ctl *__restrict__ ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        T s = 0;
        for (int32_t q = ldg(prp + i); q < ldg(prp + i + 1); q++) s += ldg(pv + q) * ldg(xc + ldg(pci + q));
        xp[i] = ldg(xpre + i) + s;
    }
}

// Down sweep fused with the restriction it feeds, one thread per coarse row
// I: t_i = p_i (b_i - sum_j a_ij xpre_j) for each member i of aggregate I
// (members in increasing index order), summed into b_c[I] (and, with PRE,
// xpre_c = dinv_c b_c). Same arithmetic, in the same order, as k_down
// followed by k_restrict; t is never stored.
template <typename T, typename TO, bool PRE, typename IDX, int U>
__global__ void __launch_bounds__(kBlock) k_down_restrict(int nc, const int32_t *__restrict__ rptr,
                                                          const int32_t *__restrict__ ridx,
                                                          const int32_t *__restrict__ sptr,
                                                          const IDX *__restrict__ col, const T *__restrict__ val,
                                                          const T *__restrict__ xpre, const T *__restrict__ b,
                                                          const T *__restrict__ p, TO *__restrict__ bc,
                                                          const T *__restrict__ dinvc, T *__restrict__ xprec,
                                                          const Ctl *__restrict__ ctl) {
    int I = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t q0 = 0, q1 = 0;
    int i = 0;
    SellRow<U, false, IDX, T> R;
    T pi = 0;
    if (I < nc) {
        q0 = ldg(rptr + I);
        q1 = ldg(rptr + I + 1);
        if (q0 < q1) {
            i = ldg(ridx + q0);
            R.load(sptr, col, val, i);
            pi = ldg(p + i);
        }
    }
    pdl_enter();
    xpre = after_wait(xpre);
    b = after_wait(b);
    ctl = after_wait(ctl);
    if (halted(ctl) || I >= nc) return;
    T sum = 0;
    for (int32_t q = q0; q < q1; q++) {
        T acc = R.dot(i, [&](int j) { return ldg(xpre + j); });
        // rounded product (never contracted into the sum), as k_down stores t
        T t = mul_rn(pi, ldg(b + i) - acc);
        sum += t;
        if (q + 1 < q1) {
            i = ldg(ridx + q + 1);
            R.load(sptr, col, val, i);
            pi = ldg(p + i);
        }
    }
    bc[I] = (TO)sum;
    if (PRE) xprec[I] = ldg(dinvc + I) * sum;
}

// Prolongation fused into the post sweep: xp_j = xpre_j + p_j x_c[agg_j] is
// formed for every gathered entry (and for the row itself), then
// z_i = xp_i + dinv_i (b_i - sum_j a_ij xp_j). Same values as k_prolong
// followed by k_post; xp is never stored.
template <typename T, typename IDX, int U>
__global__ void __launch_bounds__(kBlock) k_prolong_post(int n, const int32_t *__restrict__ sptr,
                                                         const IDX *__restrict__ col, const T *__restrict__ val,
                                                         const T *__restrict__ xpre, const T *__restrict__ p,
                                                         const int32_t *__restrict__ agg, const T *__restrict__ xc,
                                                         const T *__restrict__ b, const T *__restrict__ dinv,
                                                         T *__restrict__ z, const Ctl *__restrict__ ctl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    SellRow<U, false, IDX, T> R;
    T di = 0;
    if (i < n) {
        R.load(sptr, col, val, i);
        di = ldg(dinv + i);
    }
    pdl_enter();
    xpre = after_wait(xpre);
    xc = after_wait(xc);
    b = after_wait(b);
    ctl = after_wait(ctl);
    if (halted(ctl)) return;
    auto xp = [&](int j) {
        T x = ldg(xpre + j);
        int a = ldg(agg + j);
        if (a >= 0) x = fma_rn(ldg(p + j), ldg(xc + a), x);
        return x;
    };
    for (; i < n; i += stride) {
        T acc = R.dot(i, xp);
        z[i] = xp(i) + di * (ldg(b + i) - acc);
        if (i + stride < n) {
            R.load(sptr, col, val, i + stride);
            di = ldg(dinv + i + stride);
        }
    }
}

// ------------------------------------------------------------ hybrid Gauss-Seidel
// One sweep of the l1 hybrid Gauss-Seidel smoother (Sec. 3.1, l1 reading):
// xn = xo + M^{-1} (b - A xo), M = blockdiag(L_pp + D_l1) for FWD (rows of a
// block in increasing order) or its transpose (decreasing order). One thread
// per block of nb contiguous rows: it first copies its rows of xo into xn,
// then updates them in order, reading its own block's values from xn (the
// ones already updated) and every other block's from xo (block Jacobi).
// ZERO: xo = 0 (the first pre-smoothing sweep), x_r = d_r (b_r - acc).
// Entries are summed in storage order; with one row per block and one sweep
// the values are those of the l1-Jacobi sweeps (k_down's xpre, k_post).
template <typename T, bool FWD, bool ZERO>
__global__ void __launch_bounds__(kBlock) k_gs_sweep(int n, int nb, const int32_t *__restrict__ rp,
                                                     const int32_t *__restrict__ ci, const T *__restrict__ v,
                                                     const T *__restrict__ dinv, const T *__restrict__ b,
                                                     const T *__restrict__ xo, T *xn, const Ctl *__restrict__ ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    int64_t lo64 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * nb;
    if (lo64 >= n) return;
    const int lo = (int)lo64, hi = (int)min((int64_t)n, lo64 + nb);
    for (int r = lo; r < hi; r++) xn[r] = ZERO ? T(0) : ldg(xo + r);
    for (int q = 0; q < hi - lo; q++) {
        const int r = FWD ? lo + q : hi - 1 - q;
        T acc = 0;
        const int32_t e = ldg(rp + r + 1);
        for (int32_t k = ldg(rp + r); k < e; k++) {
            const int j = ldg(ci + k);
            T xj = (j >= lo && j < hi) ? xn[j] : (ZERO ? T(0) : ldg(xo + j));
            acc += ldg(v + k) * xj;
        }
        if (ZERO)
            xn[r] = ldg(dinv + r) * (ldg(b + r) - acc);
        else
            xn[r] = xn[r] + ldg(dinv + r) * (ldg(b + r) - acc);
    }
}

// Two-phase form of the same sweep, for blocks of at most 32 rows. Phase one,
// one thread per row over the sliced-ELL layout: acc_r = sum of a_rj x_old_j
// over every entry of row r except the in-block ones the pass has already
// updated when it reaches r (FWD: j in [lo, r); backward: j in (r, hi)),
// which contribute 0 here. Phase two, one thread per block: the recurrence
// over those entries alone (k_gs_block). Same values as k_gs_sweep up to the
// order of the sums; with one row per block the sums are k_post's.
template <typename T, typename IDX, int U, bool FWD, bool STREAM>
__global__ void __launch_bounds__(kBlock, Occ<T>::kMinBlocks) k_gs_offsum(
    int n, int nb, const int32_t *__restrict__ sptr, const IDX *__restrict__ col, const T *__restrict__ val,
    const T *__restrict__ xo, T *__restrict__ acc, const Ctl *__restrict__ ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        SELL_ROW_BEGIN
        const int lo = (i / nb) * nb, hi = min(n, lo + nb);
        T a = sell_row<U, STREAM>(c_, a_, w_, i, [&](int j) {
            bool done = FWD ? (j >= lo && j < i) : (j > i && j < hi);
            return done ? T(0) : ldg(xo + j);
        });
        acc[i] = a;
    }
}

constexpr int kGsThreads = 128;  // threads per CTA of k_gs_block (window: 33 values each)

// Phase two: one thread per block of nb <= 32 rows, rows in pass order. The
// block's new values live in a shared-memory window (33-value stride per
// thread, so threads at the same row offset use different banks);
// x_r = x_old_r + d_r (b_r - (acc_r + sum over the row's part entries of
// a_rj x_new_j)). ZERO (first pre-smoothing pass, x_old = 0): acc = 0 and
// x_r = d_r (b_r - sum).
template <typename T, bool FWD, bool ZERO>
__global__ void __launch_bounds__(kGsThreads) k_gs_block(int n, int nb, int w, const int32_t *__restrict__ pci,
                                                         const T *__restrict__ pv, const T *__restrict__ dinv,
                                                         const T *__restrict__ b, const T *__restrict__ xo,
                                                         const T *__restrict__ acc, T *__restrict__ xn,
                                                         const Ctl *__restrict__ ctl) {
    __shared__ T win[kGsThreads * 33];
    pdl_enter();
    if (halted(ctl)) return;
    int64_t lo64 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * nb;
    if (lo64 >= n) return;
    const int lo = (int)lo64, hi = (int)min((int64_t)n, lo64 + nb);
    T *wv = win + threadIdx.x * 33;
    for (int q = 0; q < hi - lo; q++) {
        const int r = FWD ? lo + q : hi - 1 - q;
        T sum = ZERO ? T(0) : ldg(acc + r);
        const int64_t e = (int64_t)r * w;
        for (int k = 0; k < w; k++) {
            const int j = ldg(pci + e + k);
            if (j >= 0) sum += ldg(pv + e + k) * wv[j - lo];
        }
        T x;
        if (ZERO)
            x = ldg(dinv + r) * (ldg(b + r) - sum);
        else
            x = ldg(xo + r) + ldg(dinv + r) * (ldg(b + r) - sum);
        wv[r - lo] = x;
        xn[r] = x;
    }
}

// Both phases of a sweep in one warp per 32-row slice, for blocks whose size
// divides 32 (so no block crosses a slice) and rows with at most kGsPart
// already-updated in-block entries. Phase one as in k_gs_offsum, one lane per
// row; phase two over the slice in 32 steps in pass order (FWD: rows
// increasing, else decreasing): at step t lane t finishes its row,
// x_t = x_old_t + d_t (b_t - acc_t), the value is broadcast by a shuffle, and
// every lane whose next in-block entry (in pass order) is column t adds
// a_rt x_t to its acc. Blocks of fewer rows run side by side in the same
// steps. Same values as k_gs_block up to the order of the sums.
constexpr int kGsPartMax = 8;

template <typename T, typename IDX, int U, bool FWD, bool ZERO, bool STREAM>
__global__ void __launch_bounds__(kBlock, Occ<T>::kMinBlocks) k_gs_warp(
    int n, int nb, int w, const int32_t *__restrict__ sptr, const IDX *__restrict__ col, const T *__restrict__ val,
    const int32_t *__restrict__ pci, const T *__restrict__ pv, const T *__restrict__ dinv, const T *__restrict__ b,
    const T *__restrict__ xo, T *__restrict__ xn, const Ctl *__restrict__ ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    const int lane = threadIdx.x & 31;
    const int nsl = (n + 31) >> 5;
    const int wstride = (int)(((int64_t)gridDim.x * blockDim.x) >> 5);
    for (int sl = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); sl < nsl; sl += wstride) {
        const int i = (sl << 5) + lane;
        const bool valid = i < n;
        T acc = 0;
        if (!ZERO && valid) {
            const int lo = (i / nb) * nb, hi = min(n, lo + nb);
            SELL_ROW_BEGIN
            acc = sell_row<U, STREAM>(c_, a_, w_, i, [&](int j) {
                bool done = FWD ? (j >= lo && j < i) : (j > i && j < hi);
                return done ? T(0) : ldg(xo + j);
            });
        }
        // the row's in-block entries in pass order (padding -1 never matches)
        int rj[kGsPartMax];
        T ra[kGsPartMax];
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < kGsPartMax; k++) {
            bool ok = valid && k < w;
            rj[k] = ok ? ldg(pci + (int64_t)i * w + k) : -1;
            ra[k] = ok ? ldg(pv + (int64_t)i * w + k) : T(0);
            cnt += rj[k] >= 0 ? 1 : 0;
        }
        int pj[kGsPartMax];
        T pa[kGsPartMax];
#pragma unroll
        for (int k = 0; k < kGsPartMax; k++) {
            if (FWD) {
                pj[k] = rj[k];
                pa[k] = ra[k];
            } else {
                pj[k] = -1;
                pa[k] = T(0);
#pragma unroll
                for (int m = 0; m < kGsPartMax; m++)
                    if (m == cnt - 1 - k) {
                        pj[k] = rj[m];
                        pa[k] = ra[m];
                    }
            }
        }
        const T bi = valid ? ldg(b + i) : T(0), di = valid ? ldg(dinv + i) : T(0);
        const T xold = (!ZERO && valid) ? ldg(xo + i) : T(0);
        T x = 0;
#pragma unroll 4
        for (int step = 0; step < 32; step++) {
            const int t = FWD ? step : 31 - step;
            if (lane == t) x = ZERO ? di * (bi - acc) : xold + di * (bi - acc);
            const T xt = __shfl_sync(0xffffffffu, x, t);
            if (pj[0] == (sl << 5) + t) {
                acc += pa[0] * xt;
#pragma unroll
                for (int k = 0; k + 1 < kGsPartMax; k++) {
                    pj[k] = pj[k + 1];
                    pa[k] = pa[k + 1];
                }
                pj[kGsPartMax - 1] = -1;
            }
        }
        if (valid) xn[i] = x;
    }
}

// Level 0 after the Gauss-Seidel post-smoothing: z = x (widened) and the
// partial sums of r.z and, for FCG(1), z.q_old. Same grid and row
// order as the level-0 k_post, so the sums are formed in the same order.
template <typename T, bool FCG>
__global__ void __launch_bounds__(kBlock, Occ<T>::kMinBlocks) k_gs_finish0(int n, const T *__restrict__ x,
                                                                           const double *__restrict__ r64,
                                                                           const double *__restrict__ qold,
                                                                           double *__restrict__ z, double *partials,
                                                                           Ctl *ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    double rz = 0.0, zq = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double zo = (double)ldg(x + i);
        z[i] = zo;
        rz += ldg(r64 + i) * zo;
        if (FCG) zq += zo * ldg(qold + i);
    }
    double sums[FCG ? 2 : 1];
    sums[0] = rz;
    if (FCG) sums[FCG ? 1 : 0] = zq;
    write_partials<FCG ? 2 : 1>(sums, partials);
}

// x_L = A_L^{-1} b_L, one warp per row; TO = float rounds the float64 result.
// UP also prolongs x_L to the next finer level.
template <typename TO, bool UP>
__global__ void __launch_bounds__(kBlock) k_coarse(int nL, const double *__restrict__ ainv,
                                                   const double *__restrict__ bL, TO *__restrict__ xL,
                                                   const Ctl *__restrict__ ctl, Up<TO> up) {
    int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    UpRow<TO> ur;
    if (UP && row < nL && lane == 0) ur.load(up, row);
    pdl_enter();
    ctl = after_wait(ctl);
    bL = after_wait(bL);
    up.xpre = after_wait(up.xpre);
    if (halted(ctl)) return;
    if (row >= nL) return;
    const double *a = ainv + (int64_t)row * nL;
    if (UP && lane == 0) ur.gather(up);
    double s = 0.0;
    for (int j = lane; j < nL; j += 32) s += ldg(a + j) * ldg(bL + j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) {
        xL[row] = (TO)s;
        if (UP) ur.store(up, row, (TO)s);
    }
}

// x = B b on the directly solved level (B: op[op_first], or the coarsest
// inverse), float64; TO = float rounds the result. W warps share a row, a lane
// takes entries lane, lane + 32 W, ... (kOpAhead of them at most: rows of up
// to 512 W entries), all loaded before the wait since B is static, so after it
// the product costs the load of b, the FMAs and the sums. Bound: the float64
// pipe, n^2 FMAs (1,036 rows: 1.7 us).
constexpr int kOpAhead = 16;
template <typename TO, bool UP, int W>
__global__ void __launch_bounds__(kBlock) k_op(int n, const double *__restrict__ B, const double *__restrict__ b,
                                               TO *__restrict__ x, const Ctl *__restrict__ ctl, Up<TO> up) {
    __shared__ double sh[kBlock / 32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, wr = w % W;
    const int row = blockIdx.x * (kBlock / 32 / W) + w / W;
    const int j0 = 32 * wr + lane;
    double v[kOpAhead];
    UpRow<TO> ur;
    if (row < n) {
        const double *a = B + (int64_t)row * n;
#pragma unroll
        for (int k = 0; k < kOpAhead; k++) v[k] = j0 + 32 * W * k < n ? ldg(a + j0 + 32 * W * k) : 0.0;
        if (UP && j0 == 0) ur.load(up, row);
    }
    pdl_enter();
    b = after_wait(b);
    ctl = after_wait(ctl);
    up.xpre = after_wait(up.xpre);
    const int halt = halted(ctl);
    double s = 0.0;
    if (row < n) {
        double bv[kOpAhead];
#pragma unroll
        for (int k = 0; k < kOpAhead; k++) bv[k] = j0 + 32 * W * k < n ? ldg(b + j0 + 32 * W * k) : 0.0;
        if (UP && j0 == 0) ur.gather(up);
#pragma unroll
        for (int k = 0; k < kOpAhead; k++)
            if (32 * W * k < n) s = fma(v[k], bv[k], s);
    }
    s = warp_sum(s);
    if (W > 1) {
        if (lane == 0) sh[w] = s;
        __syncthreads();
        if (j0 == 0)
            for (int q = 1; q < W; q++) s += sh[w + q];
    }
    if (row < n && j0 == 0 && !halt) {
        x[row] = (TO)s;
        if (UP) ur.store(up, row, (TO)s);
    }
}

// Single-level hierarchy: z = A^{-1} r (through float32 as the float32
// V-cycle would round it when F32), then r.z / z.q_old as on level 0.
template <bool F32, bool FCG>
__global__ void __launch_bounds__(kBlock) k_coarse_only(int n, const double *__restrict__ ainv,
                                                        const double *__restrict__ r, double *__restrict__ z,
                                                        const double *__restrict__ qold, double *partials,
                                                        Ctl *ctl) {
    pdl_enter();
    if (halted(ctl)) return;
    double rz = 0.0, zq = 0.0;
    int lane = threadIdx.x & 31;
    int wpb = blockDim.x >> 5;
    for (int row = blockIdx.x * wpb + (threadIdx.x >> 5); row < n; row += gridDim.x * wpb) {
        const double *a = ainv + (int64_t)row * n;
        double s = 0.0;
        for (int j = lane; j < n; j += 32) {
            double rj = ldg(r + j);
            if (F32) rj = (double)(float)rj;
            s += ldg(a + j) * rj;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) {
            double zo = F32 ? (double)(float)s : s;
            z[row] = zo;
            rz += r[row] * zo;
            if (FCG) zq += zo * qold[row];
        }
    }
    double sums[FCG ? 2 : 1];
    sums[0] = rz;
    if (FCG) sums[FCG ? 1 : 0] = zq;
    write_partials<FCG ? 2 : 1>(sums, partials);
}

// ------------------------------------------------------------ Krylov kernels
// rho = r.z and beta from the partial sums of the kernel that produced z:
// PCG beta = rho / rho_old, FCG(1) beta = -(z.q_old) / (p.q)_old (the float32
// V-cycle, and either precision when the iterative coarsest solve makes the
// V-cycle vary from one application to the next); then p = z + beta p
// (beta = 0 on a restart gives p = z). The first row's z and p and the scalars
// are requested before the partials are summed.
template <bool FCG>
__global__ void __launch_bounds__(kVecBlock) k_axpy_p(int n, const double *__restrict__ z, double *__restrict__ p,
                                                      const double *pa, int ga, Ctl *ctl) {
    pdl_enter();
    // no use of the state stands between the wait and these loads
    z = after_wait(z);
    p = after_wait(p);
    ctl = after_wait(ctl);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    int halt = kRun, restart = 0;
    double pq_old = 0.0, rho_old = 0.0;
    if (threadIdx.x == 0) {  // read once per block: block 0 may be writing (step_outcome)
        halt = halted(ctl);
        restart = state(&ctl->restart);
        pq_old = state(&ctl->pq_old);
        rho_old = state(&ctl->rho_old);
    }
    double zi = 0.0, pi = 0.0;
    if (i < n) {
        zi = z[i];
        pi = p[i];
    }
    __shared__ double sbeta;
    __shared__ bool ok;
    double sums[FCG ? 2 : 1];
    sum_partials<FCG ? 2 : 1>(pa, ga, sums);
    if (threadIdx.x == 0) {
        const double rz = sums[0], zq = FCG ? sums[FCG ? 1 : 0] : 0.0;
        const bool finite = isfinite(rz) && isfinite(zq);
        ok = halt == kRun && finite && rz > 0.0;
        sbeta = restart ? 0.0 : FCG ? -zq / pq_old : rz / rho_old;
        if (blockIdx.x == 0 && halt == kRun) {
            if (ok) {
                ctl->rho = rz;
                ctl->zq = zq;
                ctl->beta = sbeta;
            } else {
                fail(ctl, finite ? AMG_ERR_BREAKDOWN : AMG_ERR_NAN);
            }
        }
    }
    __syncthreads();
    if (!ok) return;
    const double beta = sbeta;
    for (; i < n; i += stride) {
        p[i] = zi + beta * pi;
        if (i + stride < n) {
            zi = z[i + stride];
            pi = p[i + stride];
        }
    }
}

// q = A p and the partial sums of p.q.
template <typename IDX, int U>
__global__ void __launch_bounds__(kBlock, U == kWholeRow ? 1 : 4) k_spmv(int n, const int32_t *__restrict__ sptr,
                                                    const IDX *__restrict__ col, const double *__restrict__ val,
                                                    const IDX *__restrict__ upat, const double *__restrict__ p,
                                                    double *__restrict__ q, double *partials, const Ctl *ctl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    RowOf<U, U != kWholeRow, IDX, double> R;
    if (i < n) R.load(sptr, col, val, i, upat);
    pdl_enter();
    p = after_wait(p);
    ctl = after_wait(ctl);
    const int halt = halted(ctl);
    if (U != kWholeRow && halt) return;
    double pq = 0.0;
    for (; i < n; i += stride) {
        const double pi = ldg(p + i);
        double acc = R.dot(i, [&](int j) { return ldg(p + j); });
        if (U == kWholeRow && halt) return;
        q[i] = acc;
        pq += pi * acc;
        if (i + stride < n) R.load(sptr, col, val, i + stride, upat);
    }
    double sums[1] = {pq};
    write_partials<1>(sums, partials);
}

// What the V-cycle of the mode reads besides r: FCG32 a float32 copy of r
// and xpre_0 = D_0^{-1} r in float32 (as the float32 V-cycle forms them);
// PCG64 xpre_0 = D_0^{-1} r in float64.
struct REmit {
    float *r32;
    const float *dinv32;
    float *xpre32;
    const double *dinv64;
    double *xpre64;
};

template <int MODE>
__device__ __forceinline__ void emit_r(int i, double ri, const REmit &e) {
    if (MODE == AMG_MODE_FCG32) {
        float r = (float)ri;
        e.r32[i] = r;
        e.xpre32[i] = ldg(e.dinv32 + i) * r;
    } else {
        e.xpre64[i] = ldg(e.dinv64 + i) * ri;
    }
}

// alpha = rho / p.q from the partial sums of k_spmv, then x += alpha p,
// r -= alpha q and the partial sums of ||r||^2; one thread advances the
// iteration. The first row's vectors and the scalars are requested before the
// partials are summed. BOUND: the compiler's block size. At 512 it takes 40
// registers, so that three blocks of 512 fit an SM (at 44 two do: 48 systems at
// once 198.7 ms, 196.4); at 1,024 it takes 44 and asks for the small meshes' rows
// earlier (32^3 mixed 917 us, 901).
template <int MODE, int BOUND>
__global__ void __launch_bounds__(BOUND) k_update(int n, const double *__restrict__ p,
                                                      const double *__restrict__ q, double *__restrict__ x,
                                                      double *__restrict__ r, REmit em, const double *pb, int gb,
                                                      double *partials, Ctl *ctl) {
    pdl_enter();
    p = after_wait(p);  // as in k_axpy_p
    q = after_wait(q);
    x = after_wait(x);
    r = after_wait(r);
    ctl = after_wait(ctl);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    int halt = kRun, iter = 0;
    double rho = 0.0;
    if (threadIdx.x == 0) {
        halt = halted(ctl);
        rho = state(&ctl->rho);
        iter = state(&ctl->iter);
    }
    double pi = 0.0, qi = 0.0, xi = 0.0, ro = 0.0;
    if (i < n) {
        pi = p[i];
        qi = q[i];
        xi = x[i];
        ro = r[i];
    }
    __shared__ double salpha;
    __shared__ bool ok;
    double sums[1];
    sum_partials<1>(pb, gb, sums);
    if (threadIdx.x == 0) {
        const double pq = sums[0];
        const bool finite = isfinite(pq);
        ok = halt == kRun && finite && pq > 0.0;
        salpha = rho / pq;
        if (blockIdx.x == 0 && halt == kRun) {
            if (ok) {
                ctl->pq = pq;
                ctl->alpha = salpha;
                ctl->rho_old = rho;
                ctl->pq_old = pq;
                ctl->restart = 0;
                ctl->iter = iter + 1;
            } else {
                fail(ctl, finite ? AMG_ERR_BREAKDOWN : AMG_ERR_NAN);
            }
        }
    }
    __syncthreads();
    if (!ok) return;
    const double alpha = salpha;
    double rr = 0.0;
    for (; i < n; i += stride) {
        x[i] = xi + alpha * pi;
        double ri = ro - alpha * qi;
        r[i] = ri;
        emit_r<MODE>(i, ri, em);
        rr += ri * ri;
        if (i + stride < n) {
            pi = p[i + stride];
            qi = q[i + stride];
            xi = x[i + stride];
            ro = r[i + stride];
        }
    }
    sums[0] = rr;
    write_partials<1>(sums, partials);
}

// Loop condition of the solve graph: run another body while not ended. The
// body count is bounded independently of the kernels' own bookkeeping: a body
// runs at least one iteration, so past maxit + 1 bodies the solve is ended as
// not converged.
struct Cond {
    cudaGraphConditionalHandle hc;
    int set;  // 0: not the last kernel of a graph's prefix or loop body
};

__device__ __forceinline__ void set_cond(const Cond &c, Ctl *ctl, bool body) {
    if (!c.set) return;
    if (body) {
        const int b = state(&ctl->bodies) + 1;
        ctl->bodies = b;
        if (!state(&ctl->done) && b > state(&ctl->maxit) + 1) fail(ctl, AMG_ERR_NOCONV);
    }
    cudaGraphSetConditional(c.hc, state(&ctl->done) ? 0u : 1u);
}

// r = b - A x, ||r||^2 (and ||b||^2 on INIT); also the mode's copy of r.
// INIT starts a solve. Otherwise it ends a loop body: it takes the outcome of
// the iteration before it (unless a kernel of the body has taken it), forms
// the true residual only when the recursive one met rtol, and sets the loop
// condition.
template <bool INIT, int MODE, typename IDX>
__global__ void __launch_bounds__(kBlock, 4) k_residual(int n, const int32_t *__restrict__ sptr,
                                                        const IDX *__restrict__ col,
                                                        const double *__restrict__ val, const double *__restrict__ b,
                                                        const double *__restrict__ x, double *__restrict__ r,
                                                        REmit em, const double *pc, int gc, double *partials,
                                                        Ctl *ctl, double *hist, Cond cond) {
    pdl_enter();
    b = after_wait(b);
    x = after_wait(x);
    ctl = after_wait(ctl);
    if (!INIT) {
        if (step_outcome(pc, gc, ctl, hist) != kCheck) {
            if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(cond, ctl, true);
            return;
        }
    }
    double rr = 0.0, bb = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        SELL_ROW_BEGIN
        double acc = sell_row<kUnroll, true>(c_, a_, w_, i, [&](int j) { return ldg(x + j); });
        double bi = ldg(b + i);
        double ri = bi - acc;
        r[i] = ri;
        emit_r<MODE>(i, ri, em);
        rr += ri * ri;
        if (INIT) bb += bi * bi;
    }
    double sums[2] = {rr, bb};
    if (publish_partials<2>(sums, partials, &ctl->counter)) {
        __threadfence();
        sum_partials<2>(partials, gridDim.x, sums);
        if (threadIdx.x != 0) return;
        const double a = sums[0], bsq = sums[1];
        ctl->counter = 0;
        if (INIT) {
            const double bn0 = sqrt(bsq), stop = state(&ctl->rtol) * bn0;
            ctl->bnorm = bn0;
            ctl->stop2 = stop * stop;
        }
        const double bn = state(&ctl->bnorm), rel = sqrt(a) / bn;
        if (INIT && (!isfinite(bn) || !isfinite(a))) {
            fail(ctl, AMG_ERR_NAN);
        } else if (INIT && bn == 0.0) {
            ctl->true_rel = 0.0;
            hist[0] = 0.0;
            finish(ctl);
        } else {
            ctl->true_rel = rel;
            if (INIT) ctl->rel = rel;
            if (!isfinite(rel)) {
                fail(ctl, AMG_ERR_NAN);
            } else if (rel <= state(&ctl->rtol)) {
                if (INIT) hist[0] = rel;
                finish(ctl);
            } else {
                ctl->restart = 1;
                ctl->halt = kRun;
                const int it = state(&ctl->iter);
                hist[it] = rel;
                if (it >= state(&ctl->maxit)) fail(ctl, AMG_ERR_NOCONV);
            }
        }
        set_cond(cond, ctl, !INIT);
    }
}

__global__ void k_zero(double *a, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = 0.0;
}

inline int grid_rows(int64_t n) { return (int)((n + kBlock - 1) / kBlock); }


// ------------------------------------------------------------ profiling
// CUDA-event spans around kernel launches (only when profiling is on).
// kinds: 0 down0, 1 post0 (the whole up phase of level 0 with the
// Gauss-Seidel smoother), 2 q = A p, 3 update, 4 true residual, 5 levels >= 1
// and the coarsest solve, 6 p = z + beta p, 7 prolong0.
constexpr int kEvPairs = 256;

// Opens a span of `kind` (kinds < kKinds: the kernel kinds above; kinds
// kLevelSpan + 3 l + phase: level l's down (0: down + restriction), up (1:
// prolongation + post) or coarsest (2) phase). Returns the span's slot or -1.
constexpr int kLevelSpan = 100;

int prof_begin(amg_hier *h, int kind, cudaStream_t s) {
    if (!h->profile || h->ev_used + 2 > (int)h->ev.size()) return -1;
    int slot = h->ev_used;
    h->ev_kind[slot / 2] = kind;
    cudaEventRecord(h->ev[slot], s);
    h->ev_used += 2;
    return slot;
}

void prof_end(amg_hier *h, int slot, cudaStream_t s) {
    if (slot < 0) return;
    cudaEventRecord(h->ev[slot + 1], s);
}

// Fold the recorded spans into the totals (stream already synchronised).
void prof_collect(amg_hier *h) {
    for (int k = 0; k + 1 < h->ev_used; k += 2) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, h->ev[k], h->ev[k + 1]) != cudaSuccess) continue;
        int kind = h->ev_kind[k / 2];
        if (kind >= kLevelSpan) {
            int l = (kind - kLevelSpan) / 3, ph = (kind - kLevelSpan) % 3;
            if (l < amg_hier::kMaxProfLevels) {
                h->lev_ms[l][ph] += ms;
                h->lev_n[l][ph] += 1;
            }
        } else {
            h->prof_ms[kind] += ms;
            h->prof_n[kind] += 1;
        }
    }
    h->ev_used = 0;
}

// ------------------------------------------------------------ one iteration
template <typename T>
struct LP;
template <>
struct LP<float> {
    static const float *val(const Level &l) { return l.S.v32; }
    static const float *dinv(const Level &l) { return l.dinv32; }
    static const float *p(const Level &l) { return l.p32; }
    static float *b(Level &l) { return l.b32; }
    static float *x(Level &l) { return l.x32; }
    static float *t(Level &l) { return l.t32; }
    static float *xpre(Level &l) { return l.xpre32; }
    static float *xp(Level &l) { return l.xp32; }
    static const float *r0(const amg_hier *h) { return h->r32; }
    static const float *Pv(const Level &l) { return l.P32; }
    static const float *Ptv(const Level &l) { return l.Pt32; }
    static const float *ones(const Level &l) { return l.ones32; }
    static const float *csr(const Level &l) { return l.v32csr; }
    static const float *part(const Level &l, int d) { return l.gs_v32[d]; }
    static float *acc(const Level &l) { return reinterpret_cast<float *>(l.gs_acc); }
};
template <>
struct LP<double> {
    static const double *val(const Level &l) { return l.S.v64; }
    static const double *dinv(const Level &l) { return l.dinv; }
    static const double *p(const Level &l) { return l.p; }
    static double *b(Level &l) { return l.b64; }
    static double *x(Level &l) { return l.x64; }
    static double *t(Level &l) { return l.t64; }
    static double *xpre(Level &l) { return l.xpre64; }
    static double *xp(Level &l) { return l.xp64; }
    static const double *r0(const amg_hier *h) { return h->r; }
    static const double *Pv(const Level &l) { return l.P.v; }
    static const double *Ptv(const Level &l) { return l.Pt.v; }
    static const double *ones(const Level &l) { return l.ones64; }
    static const double *csr(const Level &l) { return l.A.v; }
    static const double *part(const Level &l, int d) { return l.gs_v64[d]; }
    static double *acc(const Level &l) { return l.gs_acc; }
};

REmit remit(amg_hier *h) {
    Level &l0 = h->lev[0];
    return REmit{h->r32, l0.dinv32, l0.xpre32, l0.dinv, l0.xpre64};
}

// Launch with the level's column array: int16 offsets when present.
// BODY sees IDX (the column type), cols (the columns) and pats (the shared
// offset patterns in the column type, or null).
#define WITH_COLS(S, BODY)                          \
    do {                                            \
        if ((S).col16) {                            \
            using IDX = int16_t;                    \
            const IDX *cols = (S).col16;            \
            [[maybe_unused]] const IDX *pats = (S).upat16; \
            BODY;                                   \
        } else {                                    \
            using IDX = int32_t;                    \
            const IDX *cols = (S).col;              \
            [[maybe_unused]] const IDX *pats = (S).upat; \
            BODY;                                   \
        }                                           \
    } while (0)

template <typename T>
constexpr int prec_index() { return sizeof(T) == 4 ? 0 : 1; }

// Sections of the partial sums, 2 h->nblk values each: what k_post left for
// k_axpy_p, k_spmv for k_update, k_update for the next iteration's first
// kernel or k_residual, and k_residual's own.
inline double *parts(const amg_hier *h, int section) { return h->partials + 2 * (size_t)h->nblk * section; }
constexpr int kPartsRz = 0, kPartsPq = 1, kPartsRr = 2, kPartsTrue = 3, kPartSections = 4;

// Threads per block of a sweep with one thread per row: small levels spread
// over the SMs (4,096 rows are 64 blocks of 64 rows, not 16 of 256).
int small_block(const amg_hier *h, int n) { return n <= h->sms * 64 ? 64 : n <= h->sms * 128 ? 128 : kBlock; }

// Rows up to which a level's rows are read whole (WholeRow: one thread per
// row, ~100 registers in float32); above, 16-entry chunks keep more warps
// resident (64,512 rows: 9.9 us whole, 6.7 us in chunks).
constexpr int kWholeRows = 32768;
// A solve that shares the device (batches, serving lanes: no_tail) is short of
// registers and float64 cycles rather than waiting for latency: twelve systems
// of 24^3 to 72^3 at once ran 14.2 ms with the limits of a lone solve, 13.1
// with 1,024 and 16,384 rows (the bits are the same). In float64 the large
// systems' coarse levels lose by fusing: 48 of 24^3 to 112^3 266.3 ms with
// 16,384 rows, 263.7 with 4,096, where five small ones lose without it (24^3 to
// 41^3 2.47 ms, 2.51), so the lower limit holds for systems above 131,072 rows
// (264.6 and 2.48). In float32 twelve systems take 12.42 ms with 16,384 rows
// and 12.52 with 4,096, the 48 196.9 and 196.1.
constexpr int kWholeRowsShared = 1024;
constexpr int kFuseRowsShared = 16384, kFuseRowsLarge64 = 4096, kLargeRows64 = 131072;
int whole_rows(const amg_hier *h) { return h->no_tail ? kWholeRowsShared : kWholeRows; }

// A coarse-level sweep over n rows (or positions) in a launch shape: a thread
// per row, or without bit 1 at most one wave of the kernel's resident blocks.
template <typename... KArgs, typename... Args>
void launch_shaped(const amg_hier *h, void (*kernel)(KArgs...), int n, unsigned char shape, int blk, cudaStream_t s,
                   Args... args) {
    int g = (n + blk - 1) / blk;
    if (!(shape & 2)) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, blk, 0) != cudaSuccess || per < 1) per = 1;
        g = std::min(g, h->sms * per);
    }
    launch_k(h->pdl, kernel, g, blk, s, args...);
}
int shape_block(const amg_hier *h, int n, unsigned char shape) { return shape & 1 ? small_block(h, n) : kBlock; }

// Level l's shape of a phase (0 down, 1 up). The tuner times a shape alone;
// solves that share the device keep the fixed rule's in place of its picks (48
// systems of 24^3 to 112^3 at once 196.4 ms, 200.8 with them).
unsigned char shape_of(const amg_hier *h, int l, int pi, int phase) {
    const Level &lv = h->lev[l];
    return h->no_tail && lv.tuned[pi][phase] ? lv.rule_shape : lv.shape[pi][phase];
}

// Whether level l's down sweep can restrict in the same launch (member order),
// and whether it does: on l >= 1 only with a down shape that is not one of the
// older forms.
bool fusable(const amg_hier *h, int l, int pi) {
    const Level &lv = h->lev[l];
    const int shared = pi == 1 && h->lev[0].A.n > kLargeRows64 ? kFuseRowsLarge64 : kFuseRowsShared;
    return h->fuse && lv.mslot > 0 && !h->smoothed && !h->gs_nu && !(h->no_tail && lv.A.n > shared);
}
bool down_fused(const amg_hier *h, int l, int pi) {
    return fusable(h, l, pi) && (l == 0 || !(shape_of(h, l, pi, 0) & 12));
}

// Weight of the down sweep's output t = w (b - A xpre): the tentative
// prolongator's p (restriction by the aggregate map), or ones with
// smoothed aggregation (the restriction then applies P^T).
template <typename T>
const T *pdown(const amg_hier *h, const Level &lv) {
    return h->smoothed ? LP<T>::ones(lv) : LP<T>::p(lv);
}

// Prolongation to level l: xp = xpre + P x_{l+1} (through the aggregate map,
// or the explicit smoothed P).
template <typename T>
void launch_prolong(amg_hier *h, int l, int grid, cudaStream_t s) {
    using P = LP<T>;
    auto &lev = h->lev;
    Level &lv = lev[l];
    int n = lv.A.n;
    if (h->smoothed)
        launch_k(h->pdl, k_prolong_sa<T>, grid, kBlock, s, n, (const int32_t *)lv.P.rp, (const int32_t *)lv.P.ci,
                 P::Pv(lv), (const T *)P::xpre(lv), (const T *)P::x(lev[l + 1]), P::xp(lv), (const Ctl *)h->ctl);
    else
        launch_k(h->pdl, k_prolong<T>, grid, kBlock, s, n, (const T *)P::xpre(lv), P::p(lv), lv.agg,
                 (const T *)P::x(lev[l + 1]), P::xp(lv), (const Ctl *)h->ctl);
}

// Down sweep of level l >= 1 with the given launch shape (bits 0 and 1).
template <typename T>
void launch_down(amg_hier *h, int l, unsigned char shape, cudaStream_t s) {
    using P = LP<T>;
    Level &lv = h->lev[l];
    int n = lv.A.n;
    if (shape & 8) {
        WITH_COLS(lv.S, (launch_k(h->pdl, k_down_ml<T, IDX>, grid_rows((int64_t)n * kMlL), kBlock, s, n, lv.S.sptr,
                                  cols, P::val(lv), (const T *)P::xpre(lv), (const T *)P::b(lv), pdown<T>(h, lv),
                                  P::t(lv), (const Ctl *)h->ctl)));
        return;
    }
    const int blk = shape_block(h, n, shape);
    if ((shape & 1) && n <= whole_rows(h))
        WITH_COLS(lv.S, (launch_shaped(h, k_down<T, IDX, kWholeRow, false, false>, n, shape, blk, s, n, lv.S.sptr,
                                  cols, P::val(lv), pats, P::xpre(lv), P::b(lv), pdown<T>(h, lv), P::t(lv),
                                  (const double *)nullptr, 0, h->ctl, (double *)nullptr)));
    else if (shape & 1)
        WITH_COLS(lv.S, (launch_shaped(h, k_down<T, IDX, kUnrollSmall, false, false>, n, shape, blk, s, n,
                                  lv.S.sptr, cols, P::val(lv), pats, P::xpre(lv), P::b(lv), pdown<T>(h, lv),
                                  P::t(lv), (const double *)nullptr, 0, h->ctl, (double *)nullptr)));
    else
        WITH_COLS(lv.S, (launch_shaped(h, k_down<T, IDX, kUnroll, false, false>, n, shape, blk, s, n, lv.S.sptr, cols,
                                  P::val(lv), pats, P::xpre(lv), P::b(lv), pdown<T>(h, lv), P::t(lv),
                                  (const double *)nullptr, 0, h->ctl, (double *)nullptr)));
}

// The level whose right-hand side is float64: solved directly.
inline int direct_level(const amg_hier *h) { return h->op_first ? h->op_first : (int)h->lev.size() - 1; }

// Restriction from level l to l+1 (the directly solved one gets float64 b_L).
template <typename T>
void launch_restrict(amg_hier *h, int l, cudaStream_t s) {
    using P = LP<T>;
    auto &lev = h->lev;
    Level &lv = lev[l];
    const Ctl *ctl = h->ctl;
    if (h->smoothed) {
        if (l + 1 == direct_level(h))
            launch_k(h->pdl, k_restrict_sa<T, double, false>, grid_rows(lv.nc), kBlock, s, lv.nc,
                     (const int32_t *)lv.Pt.rp, (const int32_t *)lv.Pt.ci, P::Ptv(lv), (const T *)P::t(lv), h->bL,
                     (const T *)nullptr, (T *)nullptr, ctl);
        else
            launch_k(h->pdl, k_restrict_sa<T, T, true>, grid_rows(lv.nc), kBlock, s, lv.nc,
                     (const int32_t *)lv.Pt.rp, (const int32_t *)lv.Pt.ci, P::Ptv(lv), (const T *)P::t(lv),
                     P::b(lev[l + 1]), P::dinv(lev[l + 1]), P::xpre(lev[l + 1]), ctl);
        return;
    }
    if (l + 1 == direct_level(h))
        launch_k(h->pdl, k_restrict<T, double, false>, grid_rows(lv.nc), kBlock, s, lv.nc, lv.rptr, lv.ridx,
                 (const T *)P::t(lv), h->bL, (const T *)nullptr, (T *)nullptr, ctl);
    else
        launch_k(h->pdl, k_restrict<T, T, true>, grid_rows(lv.nc), kBlock, s, lv.nc, lv.rptr, lv.ridx,
                 (const T *)P::t(lv), P::b(lev[l + 1]), P::dinv(lev[l + 1]), P::xpre(lev[l + 1]), ctl);
}

// Level `to`'s target of a prolongation by the kernel that forms x_{to+1}.
template <typename T>
Up<T> up_of(amg_hier *h, int to) {
    using P = LP<T>;
    Level &lv = h->lev[to];
    return Up<T>{lv.mrow, lv.mslot, P::p(lv), P::xpre(lv), P::xp(lv)};
}

// Down sweep of level l with its restriction in one launch (down_fused).
template <typename T, typename TO, int U, bool STREAM, bool STEP>
void launch_down_r(amg_hier *h, int l, const T *b, TO *bc, bool pre, unsigned char shape, int blk, cudaStream_t s) {
    using P = LP<T>;
    Level &lv = h->lev[l];
    Level &nx = h->lev[l + 1];
    int lg = 0;
    while ((1 << lg) < lv.mslot) lg++;
    WITH_COLS(lv.S, (launch_shaped(h, k_down_r<T, TO, IDX, U, STREAM, STEP>, lv.mpos, shape, blk, s,
                              DownR<T, TO, IDX>{lv.mrow, lv.mpos, lv.mmain, lg, lv.S.sptr, cols, P::val(lv), pats,
                                                P::xpre(lv), b, P::p(lv), bc, pre ? P::dinv(nx) : nullptr,
                                                pre ? P::xpre(nx) : nullptr, P::xp(lv),
                                                (const double *)parts(h, kPartsRr), h->gridv, h->ctl,
                                                h->hist})));
}

// Down phase of level l >= 1: one launch in member order where the level has
// one (down_fused); else down sweep then restriction, or (shape bit 2) both in
// one launch by aggregate. Adds the kernels launched to *kernels.
template <typename T>
void launch_down_phase(amg_hier *h, int l, unsigned char shape, cudaStream_t s, int *kernels) {
    using P = LP<T>;
    if (down_fused(h, l, prec_index<T>()) && !(shape & 12)) {
        Level &lv = h->lev[l];
        const int blk = shape_block(h, lv.mpos, shape);
        const T *b = P::b(lv);
        *kernels += 1;
        if (l + 1 == direct_level(h)) {
            if ((shape & 1) && lv.A.n <= whole_rows(h))
                launch_down_r<T, double, kWholeRow, false, false>(h, l, b, h->bL, false, shape, blk, s);
            else if (shape & 1)
                launch_down_r<T, double, kUnrollSmall, false, false>(h, l, b, h->bL, false, shape, blk, s);
            else launch_down_r<T, double, kUnroll, false, false>(h, l, b, h->bL, false, shape, blk, s);
        } else {
            T *bc = P::b(h->lev[l + 1]);
            if ((shape & 1) && lv.A.n <= whole_rows(h))
                launch_down_r<T, T, kWholeRow, false, false>(h, l, b, bc, true, shape, blk, s);
            else if (shape & 1)
                launch_down_r<T, T, kUnrollSmall, false, false>(h, l, b, bc, true, shape, blk, s);
            else launch_down_r<T, T, kUnroll, false, false>(h, l, b, bc, true, shape, blk, s);
        }
        return;
    }
    *kernels += (shape & 4) && !h->smoothed ? 1 : 2;
    if (!(shape & 4) || h->smoothed) {
        launch_down<T>(h, l, shape, s);
        launch_restrict<T>(h, l, s);
        return;
    }
    auto &lev = h->lev;
    Level &lv = lev[l];
    const Ctl *ctl = h->ctl;
    int g = grid_rows(lv.nc);
    bool last = l + 1 == direct_level(h);
#define PCG_DR(U)                                                                                                   \
    do {                                                                                                            \
        if (last)                                                                                                   \
            WITH_COLS(lv.S, (launch_k(h->pdl, k_down_restrict<T, double, false, IDX, U>, g, kBlock, s, lv.nc,      \
                                      lv.rptr, lv.ridx, lv.S.sptr, cols, P::val(lv), P::xpre(lv), P::b(lv),         \
                                      P::p(lv), h->bL, (const T *)nullptr, (T *)nullptr, ctl)));                    \
        else                                                                                                        \
            WITH_COLS(lv.S, (launch_k(h->pdl, k_down_restrict<T, T, true, IDX, U>, g, kBlock, s, lv.nc, lv.rptr,   \
                                      lv.ridx, lv.S.sptr, cols, P::val(lv), P::xpre(lv), P::b(lv), P::p(lv),        \
                                      P::b(lev[l + 1]), P::dinv(lev[l + 1]), P::xpre(lev[l + 1]), ctl)));           \
    } while (0)
    if (shape & 1) PCG_DR(kUnrollSmall);
    else PCG_DR(kUnroll);
#undef PCG_DR
}

// Post sweep of level l >= 1 (z = x_l) with the given launch shape; up: it
// prolongs to level l - 1 too (not in shape 8).
template <typename T, bool UP>
void launch_post(amg_hier *h, int l, unsigned char shape, cudaStream_t s) {
    using P = LP<T>;
    Level &lv = h->lev[l];
    int n = lv.A.n;
    if (shape & 8) {
        WITH_COLS(lv.S, (launch_k(h->pdl, k_post_ml<T, IDX>, grid_rows((int64_t)n * kMlL), kBlock, s, n, lv.S.sptr,
                                  cols, P::val(lv), (const T *)P::xp(lv), (const T *)P::b(lv), P::dinv(lv), P::x(lv),
                                  (const Ctl *)h->ctl)));
        return;
    }
    const Up<T> up = UP ? up_of<T>(h, l - 1) : Up<T>{};
    const int blk = shape_block(h, n, shape);
    if ((shape & 1) && n <= whole_rows(h))
        WITH_COLS(lv.S, (launch_shaped(h, k_post<T, T, false, false, IDX, kWholeRow, false, UP>, n, shape, blk, s,
                                  n, lv.S.sptr, cols, P::val(lv), pats, P::xp(lv), P::b(lv), P::dinv(lv), P::x(lv),
                                  (const double *)nullptr, (const double *)nullptr, (double *)nullptr, h->ctl, up)));
    else if (shape & 1)
        WITH_COLS(lv.S, (launch_shaped(h, k_post<T, T, false, false, IDX, kUnrollSmall, false, UP>, n, shape, blk,
                                  s, n, lv.S.sptr, cols, P::val(lv), pats, P::xp(lv), P::b(lv), P::dinv(lv),
                                  P::x(lv), (const double *)nullptr, (const double *)nullptr, (double *)nullptr,
                                  h->ctl, up)));
    else
        WITH_COLS(lv.S, (launch_shaped(h, k_post<T, T, false, false, IDX, kUnroll, false, UP>, n, shape, blk, s, n,
                                  lv.S.sptr, cols, P::val(lv), pats, P::xp(lv), P::b(lv), P::dinv(lv), P::x(lv),
                                  (const double *)nullptr, (const double *)nullptr, (double *)nullptr, h->ctl, up)));
}

// Up phase of level l >= 1: prolongation (unless xp_ready: the kernel that
// formed x_{l+1} has done it) then post sweep, or (shape bit 2) the
// prolongation formed per gathered entry inside the post sweep. Returns
// whether it has prolonged to level l - 1 as well; adds to *kernels.
template <typename T>
bool launch_up_phase(amg_hier *h, int l, unsigned char shape, bool xp_ready, cudaStream_t s, int *kernels) {
    using P = LP<T>;
    auto &lev = h->lev;
    Level &lv = lev[l];
    int n = lv.A.n;
    const Ctl *ctl = h->ctl;
    *kernels += 1;
    if (!(shape & 4) || h->smoothed) {
        if (!xp_ready) {
            launch_prolong<T>(h, l, grid_rows(n), s);
            *kernels += 1;
        }
        if (!(shape & 8) && down_fused(h, l - 1, prec_index<T>())) {
            launch_post<T, true>(h, l, shape, s);
            return true;
        }
        launch_post<T, false>(h, l, shape, s);
        return false;
    }
    if (shape & 1)
        WITH_COLS(lv.S, (launch_shaped(h, k_prolong_post<T, IDX, kUnrollSmall>, n, shape, kBlock, s, n, lv.S.sptr,
                                  cols, P::val(lv), (const T *)P::xpre(lv), P::p(lv), lv.agg,
                                  (const T *)P::x(lev[l + 1]), (const T *)P::b(lv), P::dinv(lv), P::x(lv), ctl)));
    else
        WITH_COLS(lv.S, (launch_shaped(h, k_prolong_post<T, IDX, kUnroll>, n, shape, kBlock, s, n, lv.S.sptr, cols,
                                  P::val(lv), (const T *)P::xpre(lv), P::p(lv), lv.agg, (const T *)P::x(lev[l + 1]),
                                  (const T *)P::b(lv), P::dinv(lv), P::x(lv), ctl)));
    return false;
}

template <typename T, bool UP>
void launch_op(amg_hier *h, int D, const Up<T> &up, cudaStream_t s) {
    using P = LP<T>;
    Level &ld = h->lev[D];
    const int n = ld.A.n;
    const double *B = h->op[D] ? h->op[D] : h->Ainv;
#define PCG_OP(W)                                                                                                   \
    launch_k(h->pdl, k_op<T, UP, W>, (n + kBlock / 32 / W - 1) / (kBlock / 32 / W), kBlock, s, n, B, h->bL, P::x(ld), \
             (const Ctl *)h->ctl, up)
    if (n <= 32 * kOpAhead) PCG_OP(1);
    else if (n <= 64 * kOpAhead) PCG_OP(2);
    else if (n <= 128 * kOpAhead) PCG_OP(4);
    else PCG_OP(8);
#undef PCG_OP
}

// The directly solved level of the single-column V-cycle: x = B b with the
// explicit operator of the small levels, or x_L = A_L^{-1} b_L with the dense
// inverse, or the iterative solve (FCG + block-Jacobi ILU(1)). Adds the
// kernels launched to *kernels; *prolonged: x has been prolonged too.
template <typename T>
int launch_direct(amg_hier *h, cudaStream_t s, int *kernels, bool *prolonged) {
    using P = LP<T>;
    Level &lc = h->lev.back();
    const int D = direct_level(h);
    *prolonged = false;
    if (h->coarse_iter) {
        PCG_TRY(launch_coarse_iter<T>(h, h->cws, h->bL, P::x(lc), &h->ctl->halt, nullptr, s));
        *kernels += coarse_iter_launches(h);
        return AMG_OK;
    }
    const bool up = down_fused(h, D - 1, prec_index<T>());
    // k_op holds a row in registers ahead of the wait. In float64, where the
    // kernel before it needs the registers and the pipe, a coarsest inverse
    // above kOpMax64 rows runs faster one warp per row: per iteration 1,896 rows
    // 57.7 us with k_op and 56.3 with k_coarse, 2,285 76.2 and 66.3, 2,845 100.3
    // and 86.2, 3,906 115.7 and 109.6; in float32 45.6 and 51.8 at 1,896 rows,
    // 90.5 and 110.8 at 3,906 (62.8 and 61.7 at 2,285).
    constexpr int kOpMax64 = 1280;
    const bool whole = sizeof(T) == 4 || D + 1 < (int)h->lev.size() || h->nL <= kOpMax64;
    if (h->op_first && whole) {
        if (up) launch_op<T, true>(h, D, up_of<T>(h, D - 1), s);
        else launch_op<T, false>(h, D, Up<T>{}, s);
    } else {
        const int g = (h->nL * 32 + kBlock - 1) / kBlock;
        if (up)
            launch_k(h->pdl, k_coarse<T, true>, g, kBlock, s, h->nL, h->Ainv, h->bL, P::x(lc), (const Ctl *)h->ctl,
                     up_of<T>(h, D - 1));
        else
            launch_k(h->pdl, k_coarse<T, false>, g, kBlock, s, h->nL, h->Ainv, h->bL, P::x(lc), (const Ctl *)h->ctl,
                     Up<T>{});
    }
    *prolonged = up;
    *kernels += 1;
    return AMG_OK;
}

// One wave of the level-0 sweeps of precision T.
template <typename T>
int grid0(const amg_hier *h) { return sizeof(T) == 4 ? h->grid32 : h->grid64; }

// Float32 level-0 sweeps read whole rows at once where level 0 has shared
// offset patterns (PatRow), else 4-entry chunks.
inline bool pat_rows(const amg_hier *h) { return h->lev[0].S.upat != nullptr; }

// Level-0 down sweep t = p (b - A xpre) (evict-first matrix stream, shared
// offset patterns where level 0 has them). step: it takes the outcome of the
// iteration before it.
template <typename T, bool STEP>
void launch_down0_t(amg_hier *h, const T *b0, cudaStream_t s) {
    using P = LP<T>;
    Level &l0 = h->lev[0];
    const double *pc = parts(h, kPartsRr);
    if (down_fused(h, 0, prec_index<T>())) {
        const int blk = std::min(h->block0, small_block(h, l0.mpos));
        constexpr unsigned char shape = 2;
        T *bc = P::b(h->lev[1]);
        const bool direct = direct_level(h) == 1, whole = l0.A.n <= whole_rows(h);
        if (direct && whole) launch_down_r<T, double, kWholeRow, false, STEP>(h, 0, b0, h->bL, false, shape, blk, s);
        else if (direct) launch_down_r<T, double, kUnrollSmall, false, STEP>(h, 0, b0, h->bL, false, shape, blk, s);
        else if (whole) launch_down_r<T, T, kWholeRow, false, STEP>(h, 0, b0, bc, true, shape, blk, s);
        else launch_down_r<T, T, kUnrollSmall, false, STEP>(h, 0, b0, bc, true, shape, blk, s);
        return;
    }
    if constexpr (sizeof(T) == 4) {
        if (pat_rows(h)) {
            WITH_COLS(l0.S, (launch_k(h->pdl, k_down<T, IDX, kPatRow, true, STEP>, grid0<T>(h), h->block0, s, l0.A.n,
                                      l0.S.sptr, cols, P::val(l0), pats, (const T *)P::xpre(l0), b0,
                                      pdown<T>(h, l0), P::t(l0), pc, h->gridv, h->ctl, h->hist)));
            return;
        }
    }
    WITH_COLS(l0.S, (launch_k(h->pdl, k_down<T, IDX, kUnroll, true, STEP>, grid0<T>(h), h->block0, s, l0.A.n, l0.S.sptr,
                              cols, P::val(l0), pats, (const T *)P::xpre(l0), b0, pdown<T>(h, l0), P::t(l0), pc,
                              h->gridv, h->ctl, h->hist)));
}

template <typename T>
void launch_down0(amg_hier *h, const T *b0, bool step, cudaStream_t s) {
    if (step) launch_down0_t<T, true>(h, b0, s);
    else launch_down0_t<T, false>(h, b0, s);
}

// Level-0 post sweep z = xp + dinv (b - A xp) with r.z (and z.q_old).
template <typename T, bool FCG>
void launch_post0(amg_hier *h, const T *b0, cudaStream_t s) {
    using P = LP<T>;
    Level &l0 = h->lev[0];
    if (l0.A.n <= whole_rows(h)) {
        WITH_COLS(l0.S, (launch_k(h->pdl, k_post<T, double, true, FCG, IDX, kWholeRow, false, false>, grid0<T>(h),
                                  h->block0, s, l0.A.n, l0.S.sptr, cols, P::val(l0), pats, P::xp(l0), b0,
                                  P::dinv(l0), h->z, h->r, h->q, parts(h, kPartsRz), h->ctl, Up<T>{})));
        return;
    }
    if constexpr (sizeof(T) == 4) {
        if (pat_rows(h)) {
            WITH_COLS(l0.S, (launch_k(h->pdl, k_post<T, double, true, FCG, IDX, kPatRow, true, false>, grid0<T>(h),
                                      h->block0, s, l0.A.n, l0.S.sptr, cols, P::val(l0), pats, P::xp(l0), b0, P::dinv(l0), h->z,
                                      h->r, h->q, parts(h, kPartsRz), h->ctl,
                                      Up<T>{})));
            return;
        }
    }
    WITH_COLS(l0.S, (launch_k(h->pdl, k_post<T, double, true, FCG, IDX, kUnroll, true, false>, grid0<T>(h),
                                  h->block0, s,
                                  l0.A.n, l0.S.sptr, cols, P::val(l0), pats, P::xp(l0), b0, P::dinv(l0), h->z, h->r,
                                  h->q, parts(h, kPartsRz), h->ctl, Up<T>{})));
}

// z = B r (one V-cycle in precision T), including rho / beta. Kernels are
// launched with programmatic dependent launch when h->pdl (see pdl_enter).
template <typename T, bool FCG>
int launch_vcycle(amg_hier *h, bool step, cudaStream_t s) {
    using P = LP<T>;
    auto &lev = h->lev;
    const T *b0 = P::r0(h);
    int sp1 = prof_begin(h, 0, s);
    launch_down0<T>(h, b0, step, s);
    prof_end(h, sp1, s);
    int sp2 = prof_begin(h, 5, s);
    // levels handled by separate launches: 0..F-1; the explicit operator (or
    // the tail, or the coarsest solve) takes F..L
    int tf = h->no_tail || h->op_first ? 0 : h->tail_first[prec_index<T>()];
    int F = tf > 0 ? tf : direct_level(h);
    // per-level spans (profiling only): level l's down phase is its down
    // sweep and the restriction that leaves it (level 0: the restriction)
    int kernels = 1;  // down sweep of level 0
    for (int l = 0; l < F; l++) {
        int spl = prof_begin(h, kLevelSpan + 3 * l, s);
        unsigned char sh = shape_of(h, l, prec_index<T>(), 0);
        if (l == 0) {
            if (!down_fused(h, 0, prec_index<T>())) {
                launch_restrict<T>(h, 0, s);
                kernels += 1;
            }
        } else {
            launch_down_phase<T>(h, l, sh, s, &kernels);
        }
        prof_end(h, spl, s);
    }
    int spc = prof_begin(h, kLevelSpan + 3 * F + 2, s);
    bool xp_ready = false;
    if (tf > 0) {
        PCG_TRY(launch_smem_tail<T>(h, s));
        kernels += 1;
    } else {
        PCG_TRY(launch_direct<T>(h, s, &kernels, &xp_ready));
    }
    prof_end(h, spc, s);
    for (int l = F - 1; l >= 1; l--) {
        int spl = prof_begin(h, kLevelSpan + 3 * l + 1, s);
        xp_ready = launch_up_phase<T>(h, l, shape_of(h, l, prec_index<T>(), 1), xp_ready, s, &kernels);
        prof_end(h, spl, s);
    }
    kernels += 1;  // post sweep of level 0
    prof_end(h, sp2, s);
    if (!xp_ready) {
        int sp7 = prof_begin(h, 7, s);
        launch_prolong<T>(h, 0, h->gridp, s);
        prof_end(h, sp7, s);
        kernels += 1;
    }
    int sp3 = prof_begin(h, 1, s);
    launch_post0<T, FCG>(h, b0, s);
    prof_end(h, sp3, s);
    h->launches += kernels;
    PCG_LAUNCH_CK();
    return AMG_OK;
}

// gs_nu Gauss-Seidel sweeps on level l: pre-smoothing (forward, from zero,
// into xpre) or post-smoothing (backward, from xp, into x). Successive sweeps
// alternate between the target and t (free at both points), arranged so the
// last one writes the target. A level with a two-phase table for the pass
// (blocks of at most 32 rows) sweeps with k_gs_offsum + k_gs_block (the first
// pre-smoothing pass with k_gs_block alone); any other with k_gs_sweep.
// Returns the kernels launched.
template <typename T>
int launch_gs(amg_hier *h, int l, bool pre, const T *b, T *target, cudaStream_t s) {
    using P = LP<T>;
    Level &lv = h->lev[l];
    const int n = lv.A.n, nu = h->gs_nu, nb = gs_rows(n, h->gs_blocks);
    const unsigned g = (unsigned)((((int64_t)n + nb - 1) / nb + kBlock - 1) / kBlock);
    const Ctl *ctl = h->ctl;
    const T *src = pre ? nullptr : (const T *)P::xp(lv);
    const int d = pre ? 0 : 1;  // the forward (pre) or backward (post) pass
    // float32 only: a float64 warp instruction occupies the float64 pipe for
    // all 32 lanes, and the one-warp recurrence issues two per step with one
    // lane active; k_gs_block keeps a block per lane instead
    if (sizeof(T) == 4 && lv.gs_w[d] >= 0 && lv.gs_w[d] <= kGsPartMax && nb <= 32 && 32 % nb == 0 &&
        h->gs_fused) {
        // both phases in one launch (one warp per slice)
        const int w = lv.gs_w[d];
        const int gr = grid_rows(n);
        const bool big = n > kSmallRows;
        const int32_t *pci = lv.gs_ci[d];
        const T *pv = P::part(lv, d);
        for (int sw = 1; sw <= nu; sw++) {
            T *dst = (nu - sw) % 2 == 0 ? target : P::t(lv);
            const bool zero = pre && sw == 1;
#define PCG_GSW(UU, ST)                                                                                            \
    do {                                                                                                            \
        if (zero)                                                                                                   \
            WITH_COLS(lv.S, (launch_k(h->pdl, k_gs_warp<T, IDX, UU, true, true, ST>, gr, kBlock, s, n, nb, w,       \
                                      lv.S.sptr, cols, P::val(lv), pci, pv, P::dinv(lv), b, src, dst, ctl)));       \
        else if (pre)                                                                                               \
            WITH_COLS(lv.S, (launch_k(h->pdl, k_gs_warp<T, IDX, UU, true, false, ST>, gr, kBlock, s, n, nb, w,      \
                                      lv.S.sptr, cols, P::val(lv), pci, pv, P::dinv(lv), b, src, dst, ctl)));       \
        else                                                                                                        \
            WITH_COLS(lv.S, (launch_k(h->pdl, k_gs_warp<T, IDX, UU, false, false, ST>, gr, kBlock, s, n, nb, w,     \
                                      lv.S.sptr, cols, P::val(lv), pci, pv, P::dinv(lv), b, src, dst, ctl)));       \
    } while (0)
            if (l == 0) PCG_GSW(kUnroll, true);
            else if (big) PCG_GSW(kUnroll, false);
            else PCG_GSW(kUnrollSmall, false);
#undef PCG_GSW
            src = dst;
        }
        return nu;
    }
    if (lv.gs_w[d] >= 0) {
        // two-phase sweeps
        const int w = lv.gs_w[d];
        const unsigned gb = (unsigned)((((int64_t)n + nb - 1) / nb + kGsThreads - 1) / kGsThreads);
        const int gr = grid_rows(n);
        const bool big = n > kSmallRows;
        int kernels = 0;
        for (int sw = 1; sw <= nu; sw++) {
            T *dst = (nu - sw) % 2 == 0 ? target : P::t(lv);
            const bool zero = pre && sw == 1;
            if (!zero) {
#define PCG_OFFSUM(UU, ST)                                                                                          \
    WITH_COLS(lv.S, (launch_k(h->pdl, k_gs_offsum<T, IDX, UU, true, ST>, gr, kBlock, s, n, nb, lv.S.sptr, cols,     \
                              P::val(lv), src, P::acc(lv), ctl)))
#define PCG_OFFSUM_B(UU, ST)                                                                                        \
    WITH_COLS(lv.S, (launch_k(h->pdl, k_gs_offsum<T, IDX, UU, false, ST>, gr, kBlock, s, n, nb, lv.S.sptr, cols,    \
                              P::val(lv), src, P::acc(lv), ctl)))
                if (pre) {
                    if (l == 0) PCG_OFFSUM(kUnroll, true);
                    else if (big) PCG_OFFSUM(kUnroll, false);
                    else PCG_OFFSUM(kUnrollSmall, false);
                } else {
                    if (l == 0) PCG_OFFSUM_B(kUnroll, true);
                    else if (big) PCG_OFFSUM_B(kUnroll, false);
                    else PCG_OFFSUM_B(kUnrollSmall, false);
                }
#undef PCG_OFFSUM
#undef PCG_OFFSUM_B
                kernels++;
            }
            const int32_t *pci = lv.gs_ci[d];
            const T *pv = P::part(lv, d);
            if (zero)
                launch_k(h->pdl, k_gs_block<T, true, true>, gb, kGsThreads, s, n, nb, w, pci, pv, P::dinv(lv), b,
                         (const T *)nullptr, (const T *)nullptr, dst, ctl);
            else if (pre)
                launch_k(h->pdl, k_gs_block<T, true, false>, gb, kGsThreads, s, n, nb, w, pci, pv, P::dinv(lv), b,
                         src, (const T *)P::acc(lv), dst, ctl);
            else
                launch_k(h->pdl, k_gs_block<T, false, false>, gb, kGsThreads, s, n, nb, w, pci, pv, P::dinv(lv), b,
                         src, (const T *)P::acc(lv), dst, ctl);
            kernels++;
            src = dst;
        }
        return kernels;
    }
    for (int sw = 1; sw <= nu; sw++) {
        T *dst = (nu - sw) % 2 == 0 ? target : P::t(lv);
        if (pre && sw == 1)
            launch_k(h->pdl, k_gs_sweep<T, true, true>, g, kBlock, s, n, nb, (const int32_t *)lv.A.rp,
                     (const int32_t *)lv.A.ci, P::csr(lv), P::dinv(lv), b, (const T *)nullptr, dst, ctl);
        else if (pre)
            launch_k(h->pdl, k_gs_sweep<T, true, false>, g, kBlock, s, n, nb, (const int32_t *)lv.A.rp,
                     (const int32_t *)lv.A.ci, P::csr(lv), P::dinv(lv), b, src, dst, ctl);
        else
            launch_k(h->pdl, k_gs_sweep<T, false, false>, g, kBlock, s, n, nb, (const int32_t *)lv.A.rp,
                     (const int32_t *)lv.A.ci, P::csr(lv), P::dinv(lv), b, src, dst, ctl);
        src = dst;
    }
    return nu;
}

// z = B r with the hybrid Gauss-Seidel smoother (gs_nu sweeps each side):
// the l1-Jacobi V-cycle with its smoothing steps replaced, the coarsest solve
// by launch_coarsest (no cluster tail), rho and beta by k_gs_finish0.
template <typename T, bool FCG>
int launch_vcycle_gs(amg_hier *h, cudaStream_t s) {
    using P = LP<T>;
    auto &lev = h->lev;
    const int L = direct_level(h);  // smoothed levels: 0..L-1
    Ctl *ctl = h->ctl;
    Level &l0 = lev[0];
    const T *b0 = P::r0(h);
    const bool pdl = h->pdl;
    int kernels = 0;
    int sp1 = prof_begin(h, 0, s);
    kernels += launch_gs<T>(h, 0, true, b0, P::xpre(l0), s);
    launch_down0<T>(h, b0, false, s);
    kernels += 1;
    prof_end(h, sp1, s);
    int sp2 = prof_begin(h, 5, s);
    for (int l = 0; l < L; l++) {
        int spl = prof_begin(h, kLevelSpan + 3 * l, s);
        unsigned char sh = shape_of(h, l, prec_index<T>(), 0);
        if (l == 0) {
            launch_restrict<T>(h, 0, s);
            kernels += 1;
        } else {
            kernels += launch_gs<T>(h, l, true, P::b(lev[l]), P::xpre(lev[l]), s);
            launch_down_phase<T>(h, l, sh, s, &kernels);
        }
        prof_end(h, spl, s);
    }
    int spc = prof_begin(h, kLevelSpan + 3 * L + 2, s);
    bool prolonged = false;
    PCG_TRY(launch_direct<T>(h, s, &kernels, &prolonged));
    prof_end(h, spc, s);
    for (int l = L - 1; l >= 1; l--) {
        Level &lv = lev[l];
        int spl = prof_begin(h, kLevelSpan + 3 * l + 1, s);
        launch_prolong<T>(h, l, grid_rows(lv.A.n), s);
        kernels += 1 + launch_gs<T>(h, l, false, P::b(lv), P::x(lv), s);
        prof_end(h, spl, s);
    }
    prof_end(h, sp2, s);
    int sp3 = prof_begin(h, 1, s);
    launch_prolong<T>(h, 0, h->gridp, s);
    kernels += 1 + launch_gs<T>(h, 0, false, b0, P::x(l0), s);
    // the post sweep's grid, so rho is summed in the same order as there
    launch_k(pdl, k_gs_finish0<T, FCG>, grid0<T>(h), h->block0, s, l0.A.n, (const T *)P::x(l0), (const double *)h->r,
             (const double *)h->q, h->z, parts(h, kPartsRz), ctl);
    kernels += 1;
    prof_end(h, sp3, s);
    h->launches += kernels;
    PCG_LAUNCH_CK();
    return AMG_OK;
}

// One iteration. first / last: its place in a loop body (or in a chunk of
// stream launches); cond is set by the body's last kernel. An l1-Jacobi
// V-cycle's first kernel takes the outcome of the iteration before it in the
// body, so only the body's last iteration launches k_residual (one launch per
// iteration less: 2.5 us); the other V-cycles launch it after every iteration.
template <int MODE>
int launch_iteration_t(amg_hier *h, bool first, bool last, const Cond &cond, cudaStream_t s) {
    int L = (int)h->lev.size() - 1;
    Level &l0 = h->lev[0];
    int n = l0.A.n;
    const bool pdl = h->pdl;
    const bool takes = L > 0 && !h->gs_nu;  // the V-cycle can take an outcome
    const bool step = takes && !first;
    int ga = MODE == AMG_MODE_FCG32 ? h->grid32 : h->grid64;  // blocks of the kernel that left r.z
    if (L == 0) {
        ga = h->gridv;
        launch_k(pdl, k_coarse_only<MODE == AMG_MODE_FCG32, MODE == AMG_MODE_FCG32>, h->gridv, kBlock, s, h->nL,
                 h->Ainv, h->r, h->z, h->q, parts(h, kPartsRz), h->ctl);
        h->launches += 1;
    } else if (MODE == AMG_MODE_FCG32) {
        if (h->gs_nu) PCG_TRY((launch_vcycle_gs<float, true>(h, s)));
        else PCG_TRY((launch_vcycle<float, true>(h, step, s)));
    } else if (h->coarse_iter) {
        // the float64 V-cycle is not a fixed operator either: FCG(1) beta
        if (h->gs_nu) PCG_TRY((launch_vcycle_gs<double, true>(h, s)));
        else PCG_TRY((launch_vcycle<double, true>(h, step, s)));
    } else {
        if (h->gs_nu) PCG_TRY((launch_vcycle_gs<double, false>(h, s)));
        else PCG_TRY((launch_vcycle<double, false>(h, step, s)));
    }
    int sp4 = prof_begin(h, 6, s);
    if (MODE == AMG_MODE_FCG32 || h->coarse_iter)
        launch_k(pdl, k_axpy_p<true>, h->gridv, h->blockv, s, n, h->z, h->p, parts(h, kPartsRz), ga, h->ctl);
    else
        launch_k(pdl, k_axpy_p<false>, h->gridv, h->blockv, s, n, h->z, h->p, parts(h, kPartsRz), ga, h->ctl);
    prof_end(h, sp4, s);
    int sp5 = prof_begin(h, 2, s);
    if (n <= whole_rows(h))
        WITH_COLS(l0.S, (launch_k(pdl, k_spmv<IDX, kWholeRow>, h->grid64, h->block0, s, n, l0.S.sptr, cols, l0.S.v64,
                                  pats, h->p, h->q, parts(h, kPartsPq), h->ctl)));
    else
        WITH_COLS(l0.S, (launch_k(pdl, k_spmv<IDX, kUnroll>, h->grid64, h->block0, s, n, l0.S.sptr, cols, l0.S.v64,
                                  pats, h->p, h->q, parts(h, kPartsPq), h->ctl)));
    prof_end(h, sp5, s);
    int sp6 = prof_begin(h, 3, s);
    if (h->vec_per_sm == 2)
        launch_k(pdl, k_update<MODE, 2 * kVecBlock>, h->gridv, h->blockv, s, n, h->p, h->q, h->x, h->r, remit(h),
                 parts(h, kPartsPq), h->grid64, parts(h, kPartsRr), h->ctl);
    else
        launch_k(pdl, k_update<MODE, kVecBlock>, h->gridv, h->blockv, s, n, h->p, h->q, h->x, h->r, remit(h),
                 parts(h, kPartsPq), h->grid64, parts(h, kPartsRr), h->ctl);
    prof_end(h, sp6, s);
    h->launches += 3;
    if (last || !takes) {
        int sp7 = prof_begin(h, 4, s);
        WITH_COLS(l0.S, (launch_k(pdl, k_residual<false, MODE, IDX>, h->grid64, h->block0, s, n, l0.S.sptr, cols,
                                  l0.S.v64, h->b, h->x, h->r, remit(h), parts(h, kPartsRr), h->gridv,
                                  parts(h, kPartsTrue), h->ctl, h->hist, last ? cond : Cond{})));
        prof_end(h, sp7, s);
        h->launches += 1;
    }
    PCG_LAUNCH_CK();
    return AMG_OK;
}

int launch_iteration(amg_hier *h, bool first, bool last, const Cond &cond, cudaStream_t s) {
    if (h->mode == AMG_MODE_FCG32) return launch_iteration_t<AMG_MODE_FCG32>(h, first, last, cond, s);
    return launch_iteration_t<AMG_MODE_PCG64>(h, first, last, cond, s);
}

int launch_prefix(amg_hier *h, const Cond &cond, cudaStream_t s) {
    Level &l0 = h->lev[0];
    int n = l0.A.n;
    k_zero<<<grid_rows(n), kBlock, 0, s>>>(h->p, n);
    k_zero<<<grid_rows(n), kBlock, 0, s>>>(h->q, n);
    if (h->mode == AMG_MODE_FCG32)
        WITH_COLS(l0.S, (launch_k(h->pdl, k_residual<true, AMG_MODE_FCG32, IDX>, h->grid64, h->block0, s, n, l0.S.sptr,
                                  cols, l0.S.v64, h->b, h->x, h->r, remit(h), (const double *)nullptr, 0,
                                  parts(h, kPartsTrue), h->ctl, h->hist, cond)));
    else
        WITH_COLS(l0.S, (launch_k(h->pdl, k_residual<true, AMG_MODE_PCG64, IDX>, h->grid64, h->block0, s, n, l0.S.sptr,
                                  cols, l0.S.v64, h->b, h->x, h->r, remit(h), (const double *)nullptr, 0,
                                  parts(h, kPartsTrue), h->ctl, h->hist, cond)));
    h->launches += 3;
    PCG_LAUNCH_CK();
    return AMG_OK;
}

}  // namespace

// Captures the prefix of one whole solve of h in `mode` onto cs, which must
// be capturing (possibly as a forked branch of a larger capture): zero p/q,
// first residual (which sets the loop condition), and a while node whose body is
// filled later by capture_solve_body. Kernel counts go to *prefix_k.
int capture_solve_prefix(amg_hier *h, int mode, cudaStream_t cs, PendingBody *pb, int *prefix_k) {
    int saved_mode = h->mode;
    h->mode = mode;
    int64_t l0 = h->launches;
    int st = AMG_OK;
    cudaGraph_t g = nullptr;
    cudaGraphConditionalHandle hc = 0;
    cudaStreamCaptureStatus cst;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    cudaGraphNodeParams cp = {};
    cudaGraphNode_t cnode = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, &g, nullptr, nullptr, nullptr);
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&hc, g, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) st = launch_prefix(h, Cond{hc, 1}, cs);
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
    *prefix_k = (int)(h->launches - l0);
    h->launches = l0;
    h->mode = saved_mode;
    if (st) return st;
    if (e != cudaSuccess) return cuda_fail(e, "solve graph capture", __FILE__, __LINE__);
    pb->h = h;
    pb->mode = mode;
    pb->body = cp.conditional.phGraph_out[0];
    pb->hc = hc;
    return AMG_OK;
}

// Fills the while node's body: kBodyIters iterations, the last kernel of which
// sets the loop condition, captured on s (not capturing). Kernel count of one
// body to *body_k.
constexpr int kBodyIters = 4;
int capture_solve_body(const PendingBody &pb, cudaStream_t s, int *body_k) {
    amg_hier *h = pb.h;
    int saved_mode = h->mode;
    h->mode = pb.mode;
    int64_t l1 = h->launches;
    int st = AMG_OK;
    cudaError_t e = cudaStreamBeginCaptureToGraph(s, pb.body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int k = 0; k < kBodyIters && !st; k++)
            st = launch_iteration(h, k == 0, k + 1 == kBodyIters, Cond{pb.hc, 1}, s);
        cudaGraph_t bout = pb.body;
        cudaError_t e2 = cudaStreamEndCapture(s, &bout);
        if (e2 != cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    *body_k = (int)(h->launches - l1);
    h->launches = l1;
    h->mode = saved_mode;
    if (st) return st;
    if (e != cudaSuccess) return cuda_fail(e, "solve graph body capture", __FILE__, __LINE__);
    return AMG_OK;
}

namespace {

// Whole solve as one graph: prefix (zero p/q, first residual), then a while
// node whose body is kBodyIters iterations.
// tail = false builds the variant without the shared-memory tail.
int build_graph(amg_hier *h, int mode, bool tail = true) {
    if (!h->cap_stream) PCG_CK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    cudaStream_t cs = h->cap_stream;
    PendingBody pb;
    int prefix = 0, body_k = 0;
    cudaGraphExec_t &exec = tail ? h->gexec[mode] : h->gexec_nt[mode];
    h->no_tail = tail ? 0 : 1;
    PCG_CK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    int st = capture_solve_prefix(h, mode, cs, &pb, &prefix);
    cudaGraph_t full = nullptr;
    cudaError_t e = cudaStreamEndCapture(cs, &full);
    if (!st && e != cudaSuccess) st = cuda_fail(e, "solve graph capture", __FILE__, __LINE__);
    if (!st) st = capture_solve_body(pb, cs, &body_k);
    h->no_tail = 0;
    if (st) {
        if (full) cudaGraphDestroy(full);
        return st;
    }
    e = cudaGraphInstantiate(&exec, full, 0);
    cudaGraphDestroy(full);
    if (e != cudaSuccess) {
        exec = nullptr;
        return cuda_fail(e, "cudaGraphInstantiate", __FILE__, __LINE__);
    }
    h->graph_prefix_kernels = prefix;
    (tail ? h->graph_body_kernels : h->graph_body_kernels_nt)[mode] = body_k;
    return AMG_OK;
}

bool is_device_ptr(const void *p) {
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

// Shared-memory cluster tail (tail.cu) of a handle without the explicit
// operator. PCGAMG_TAIL=0: no tail and no transfers inside the sweeps, every
// sweep and transfer of the levels above the directly solved one its own launch.
int setup_tail(amg_hier *h) {
    h->tail_first[0] = h->tail_first[1] = 0;
    const char *e = getenv("PCGAMG_TAIL");
    if (e && e[0] == '0') {
        h->fuse = 0;
        return AMG_OK;
    }
    // the tail holds a dense coarsest inverse and aggregate-map transfers
    if (h->coarse_iter || h->smoothed || h->op_first) return AMG_OK;
    return setup_smem_tail(h);
}

int set_profile(amg_hier *h, int enable) {
    if (enable && h->ev.empty()) {
        h->ev.resize(2 * kEvPairs);
        for (auto &e : h->ev) PCG_CK(cudaEventCreate(&e));
    }
    h->profile = enable ? 1 : 0;
    h->ev_used = 0;
    return AMG_OK;
}

void free_profile(amg_hier *h) {
    for (auto &e : h->ev) cudaEventDestroy(e);
    h->ev.clear();
    drop_graphs(h);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    h->cap_stream = nullptr;
}

int alloc_solve_workspace(amg_hier *h) {
    Mem &M = h->mem;
    int n = h->lev[0].A.n;
    int dev = 0, sms = 0;
    PCG_CK(cudaGetDevice(&dev));
    PCG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    h->device = dev;
    h->sms = sms;
    // One wave of resident blocks per level-0 kernel family (grid = SMs x
    // blocks resident per SM), capped by the rows available.
    // A mesh of less than a full block per SM takes smaller blocks, one per SM.
    h->block0 = std::min(kBlock, std::max(64, ((n + sms - 1) / sms + 31) / 32 * 32));
    auto wave = [&](const void *fn, int *grid) -> int {
        int per = 0;
        PCG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, h->block0, 0));
        int64_t want = ((int64_t)n + h->block0 - 1) / h->block0;
        int64_t g = (int64_t)sms * (per > 0 ? per : 1);
        *grid = (int)(want < g ? want : g);
        if (*grid < 1) *grid = 1;
        return AMG_OK;
    };
    PCG_TRY(wave((const void *)k_down<float, int32_t, kUnroll, true, true>, &h->grid32));
    if (pat_rows(h)) {
        // the whole-row sweeps: one wave of the fewer of their resident blocks
        int gd = 0, gp = 0;
        if (h->lev[0].S.col16) {
            PCG_TRY(wave((const void *)k_down<float, int16_t, kPatRow, true, true>, &gd));
            PCG_TRY(wave((const void *)k_post<float, double, true, true, int16_t, kPatRow, true, false>, &gp));
        } else {
            PCG_TRY(wave((const void *)k_down<float, int32_t, kPatRow, true, true>, &gd));
            PCG_TRY(wave((const void *)k_post<float, double, true, true, int32_t, kPatRow, true, false>, &gp));
        }
        h->grid32 = std::min(gd, gp);
    }
    PCG_TRY(wave((const void *)k_spmv<int32_t, kUnroll>, &h->grid64));
    PCG_TRY(wave((const void *)k_prolong<float>, &h->gridp));
    // the vector kernels: few blocks (their consumers read one partial per
    // block), the block as large as the rows fill. Two per SM while they hold
    // the rows (41^3 float64 2,242 us with three, 2,183 with two), three above
    // (64^3 warm 2,155 and 2,136). Blocks of 1,024 threads, two per SM, waited
    // for half an SM to fall free where systems share the device: 48 of 24^3 to
    // 112^3 at once 203.8 ms (196.1 with three blocks of 512).
    h->vec_per_sm = n <= 2 * sms * kVecBlock ? 2 : 3;
    const int vec_blocks = h->vec_per_sm * sms;
    h->blockv = (int)std::min<int64_t>(kVecBlock, std::max<int64_t>(128, ((int64_t)n + vec_blocks - 1) / vec_blocks));
    h->blockv = (h->blockv + 31) / 32 * 32;
    h->gridv = std::min(vec_blocks, (n + h->blockv - 1) / h->blockv);
    h->nblk = std::max(h->grid32, std::max(h->grid64, h->gridv));
    // the coarse levels' fixed shape rule
    for (size_t l = 1; l < h->lev.size(); l++) {
        unsigned char d = (unsigned char)((h->lev[l].A.n <= kSmallRows ? 1 : 0) | 2);
        h->lev[l].rule_shape = d;
        for (auto &pr : h->lev[l].shape) pr[0] = pr[1] = d;
    }
    PCG_TRY(alloc(M, &h->b, n));
    PCG_TRY(alloc(M, &h->x, n));
    PCG_TRY(alloc(M, &h->r, n));
    PCG_TRY(alloc(M, &h->r32, n));
    PCG_TRY(alloc(M, &h->z, n));
    PCG_TRY(alloc(M, &h->q, n));
    PCG_TRY(alloc(M, &h->p, n));
    PCG_TRY(alloc(M, &h->partials, 2 * (size_t)h->nblk * kPartSections));
    PCG_TRY(alloc(M, &h->ctl, 1));
    PCG_CK(cudaMemsetAsync(h->ctl, 0, sizeof(Ctl), M.stream));
    PCG_CK(cudaMallocHost(&h->ctl_host, sizeof(Ctl)));
    h->hist_cap = 1001;
    PCG_TRY(alloc(M, &h->hist, h->hist_cap));
    if (h->coarse_iter) PCG_TRY(cws_alloc(h, M, h->cws, 1));
    PCG_TRY(ops_alloc(h));
    PCG_TRY(setup_tail(h));
    return AMG_OK;
}

// Launch-shape tuner: for every swept level l >= 1, from the coarsest up, each
// V-cycle precision and each phase (down: down sweep + restriction; up:
// prolongation + post sweep), times the nine shapes (4- or 16-entry chunks x
// one-wave or one-thread-per-row grid x separate sweeps and transfers or those
// fused by aggregate; rows by four lanes) on this device, `reps` runs each
// after one warm-up run, and moves to the fastest only if it beats the current
// shape by more than 3% (so timing noise does not flip shapes). A candidate is
// timed as it would run: it is the level's shape meanwhile, as that decides
// which transfers are fused, and a prolongation that it leaves to a launch of
// its own where another candidate would not is timed with it. Work vectors are
// zeroed first; the inputs only set the timing. Captured solve graphs are
// dropped.
constexpr int kShapes = 9;  // 0..7, and 8: multi-lane rows

// Whether the kernel that forms x_{l+1} prolongs it to a level l that is fused.
template <typename T>
bool below_prolongs(const amg_hier *h, int l) {
    const int pi = prec_index<T>();
    const int tf = h->no_tail || h->op_first ? 0 : h->tail_first[pi];
    if (l + 1 >= (tf > 0 ? tf : direct_level(h))) return tf == 0 && !h->coarse_iter;
    return !(h->lev[l + 1].shape[pi][1] & 12);
}

// One run of a level's down (sweep = 0) or up phase with its current shapes
// (an up shape with bit 2 takes no prolongation).
template <typename T>
void run_phase(amg_hier *h, int l, int sweep, cudaStream_t s) {
    const int pi = prec_index<T>();
    const unsigned char *sh = h->lev[l].shape[pi];
    const bool ready = down_fused(h, l, pi) && below_prolongs<T>(h, l);
    int kernels = 0;
    if (sweep == 0) {
        launch_down_phase<T>(h, l, sh[0], s, &kernels);
        if (!ready && fusable(h, l, pi) && below_prolongs<T>(h, l) && !(sh[1] & 4)) {
            launch_prolong<T>(h, l, grid_rows(h->lev[l].A.n), s);
            kernels += 1;
        }
    } else if (!launch_up_phase<T>(h, l, sh[1], ready, s, &kernels) && down_fused(h, l - 1, pi) &&
               (l == 1 || !(h->lev[l - 1].shape[pi][1] & 4))) {
        launch_prolong<T>(h, l - 1, l == 1 ? h->gridp : grid_rows(h->lev[l - 1].A.n), s);
        kernels += 1;
    }
    h->launches += kernels;
}

template <typename T>
int tune_level(amg_hier *h, int l, cudaStream_t s, int reps, cudaEvent_t e0, cudaEvent_t e1, int *changed) {
    const int pi = prec_index<T>();
    for (int sweep = 0; sweep < 2; sweep++) {
        unsigned char &shape = h->lev[l].shape[pi][sweep];
        const unsigned char had = shape;
        float best = 0.0f, cur = 0.0f;
        int pick = -1;
        cudaError_t e = cudaSuccess;
        for (int c = 0; c < kShapes && e == cudaSuccess; c++) {
            shape = (unsigned char)c;
            run_phase<T>(h, l, sweep, s);
            e = cudaEventRecord(e0, s);
            for (int r = 0; r < reps; r++) run_phase<T>(h, l, sweep, s);
            if (e == cudaSuccess) e = cudaEventRecord(e1, s);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaGetLastError();
            float ms = 0.0f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (c == had) cur = ms;
            if (pick < 0 || ms < best) {
                best = ms;
                pick = c;
            }
        }
        shape = had;
        PCG_CK(e);
        if (best <= 0.97f * cur && pick != had) {
            shape = (unsigned char)pick;
            h->lev[l].tuned[pi][sweep] = true;
            (*changed)++;
        }
    }
    return AMG_OK;
}

int autotune_impl(amg_hier *h, cudaStream_t s, int reps, int *changed) {
    int L = (int)h->lev.size() - 1;
    *changed = 0;
    // the shapes tune the l1-Jacobi sweeps and the tentative transfers only
    if (h->gs_nu || h->smoothed) return AMG_OK;
    if (reps < 1) reps = 1;
    PCG_CK(cudaMemsetAsync(h->ctl, 0, sizeof(Ctl), s));
    for (int l = 1; l <= L; l++) {
        Level &lv = h->lev[l];
        size_t n = (size_t)lv.A.n;
        for (float *v : {lv.b32, lv.x32, lv.t32, lv.xpre32, lv.xp32})
            if (v) PCG_CK(cudaMemsetAsync(v, 0, n * sizeof(float), s));
        for (double *v : {lv.b64, lv.x64, lv.t64, lv.xpre64, lv.xp64})
            if (v) PCG_CK(cudaMemsetAsync(v, 0, n * sizeof(double), s));
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int st = AMG_OK;
    cudaError_t ce = cudaEventCreate(&e0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e1);
    if (ce != cudaSuccess) st = cuda_fail(ce, "autotune events", __FILE__, __LINE__);
    for (int l = direct_level(h) - 1; l >= 1 && !st; l--) {
        st = tune_level<float>(h, l, s, reps, e0, e1, changed);
        if (!st) st = tune_level<double>(h, l, s, reps, e0, e1, changed);
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    drop_graphs(h);
    PCG_CK(cudaStreamSynchronize(s));
    return st;
}

// Drops every captured whole-solve graph of h (they are rebuilt on the next
// solve) and marks batch graphs holding h as stale.
void drop_graphs(amg_hier *h) {
    for (auto *set : {h->gexec, h->gexec_nt, h->multi.gexec})
        for (int m = 0; m < 2; m++) {
            if (set[m]) cudaGraphExecDestroy(set[m]);
            set[m] = nullptr;
        }
    h->graph_gen++;
}

// Makes room for maxit+1 history values (invalidates captured graphs).
int ensure_hist(amg_hier *h, int maxit) {
    if (maxit + 1 <= h->hist_cap) return AMG_OK;
    release(h->mem, h->hist);
    h->hist_cap = maxit + 1;
    PCG_TRY(alloc(h->mem, &h->hist, h->hist_cap));
    drop_graphs(h);
    return AMG_OK;
}

// Serving lane. solve_prepare makes the whole-solve graph of `mode` (and a
// history of maxit + 1) ready; solve_launch starts one solve on s without
// waiting (b, x0: host or device, copied into h's own vectors) and copies the
// final state to the pinned mirror; once s has passed it, solve_collect
// writes x (host or device; zeros when b = 0) and the outcome.
int solve_prepare(amg_hier *h, int mode, int maxit) {
    PCG_TRY(ensure_hist(h, maxit));
    if (!h->gexec_nt[mode]) PCG_TRY(build_graph(h, mode, false));
    return AMG_OK;
}

int solve_launch(amg_hier *h, int mode, const double *b, const double *x0, double rtol, int maxit, cudaStream_t s) {
    int n = h->lev[0].A.n;
    h->mem.stream = s;
    PCG_TRY(solve_prepare(h, mode, maxit));
    PCG_CK(cudaMemcpyAsync(h->b, b, sizeof(double) * n, cudaMemcpyDefault, s));
    PCG_CK(cudaMemcpyAsync(h->x, x0, sizeof(double) * n, cudaMemcpyDefault, s));
    Ctl c0;
    memset(&c0, 0, sizeof(c0));
    c0.rtol = rtol;
    c0.maxit = maxit;
    c0.mode = mode;
    c0.flex = h->coarse_iter;
    c0.restart = 1;
    *h->ctl_host = c0;
    PCG_CK(cudaMemcpyAsync(h->ctl, h->ctl_host, sizeof(Ctl), cudaMemcpyHostToDevice, s));
    PCG_CK(cudaGraphLaunch(h->gexec_nt[mode], s));
    PCG_CK(cudaMemcpyAsync(h->ctl_host, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    return AMG_OK;
}

int solve_collect(amg_hier *h, int mode, double *x, cudaStream_t s, int *status, int *iters, double *true_rel,
                  int64_t *kernels) {
    int n = h->lev[0].A.n;
    const Ctl &c = *h->ctl_host;
    if (c.done == 1 && c.bnorm == 0.0) {
        k_zero<<<grid_rows(n), kBlock, 0, s>>>(h->x, n);
        PCG_LAUNCH_CK();
    }
    PCG_CK(cudaMemcpyAsync(x, h->x, sizeof(double) * n, cudaMemcpyDefault, s));
    int64_t k = h->graph_prefix_kernels + (int64_t)c.bodies * h->graph_body_kernels_nt[mode];
    h->launches += k;
    if (kernels) *kernels = k;
    if (status) *status = c.done ? c.status : AMG_ERR_NOCONV;
    if (iters) *iters = c.iter;
    if (true_rel) *true_rel = c.true_rel;
    h->last_true_rel = c.true_rel;
    return AMG_OK;
}

int solve_impl(amg_hier *h, const double *b, double *x, double rtol, int maxit, int *iters, double *res_hist,
               cudaStream_t s) {
    if (!b || !x || !(rtol >= 0.0) || maxit < 0) {
        set_error("pcg_solve: bad arguments");
        return AMG_ERR_ARG;
    }
    Level &l0 = h->lev[0];
    int n = l0.A.n;
    h->mem.stream = s;
    if (maxit + 1 > h->hist_cap) {
        release(h->mem, h->hist);
        h->hist_cap = maxit + 1;
        PCG_TRY(alloc(h->mem, &h->hist, h->hist_cap));
        drop_graphs(h);
    }
    bool bdev = is_device_ptr(b), xdev = is_device_ptr(x);
    PCG_CK(cudaMemcpyAsync(h->b, b, sizeof(double) * n, bdev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    PCG_CK(cudaMemcpyAsync(h->x, x, sizeof(double) * n, xdev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    Ctl c0;
    memset(&c0, 0, sizeof(c0));
    c0.rtol = rtol;
    c0.maxit = maxit;
    c0.mode = h->mode;
    c0.flex = h->coarse_iter;
    c0.restart = 1;
    *h->ctl_host = c0;
    PCG_CK(cudaMemcpyAsync(h->ctl, h->ctl_host, sizeof(Ctl), cudaMemcpyHostToDevice, s));
    bool graph = h->use_graph && !h->profile;
    if (graph && !h->gexec[h->mode]) {
        if (build_graph(h, h->mode) != AMG_OK) {
            h->use_graph = 0;  // keep solving with stream launches; the reason stays in amg_last_error
            graph = false;
        }
    }
    if (graph) {
        PCG_CK(cudaGraphLaunch(h->gexec[h->mode], s));
        PCG_CK(cudaMemcpyAsync(h->ctl_host, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
        PCG_CK(cudaStreamSynchronize(s));
        h->launches += h->graph_prefix_kernels + (int64_t)h->ctl_host->bodies * h->graph_body_kernels[h->mode];
    } else {
        PCG_TRY(launch_prefix(h, Cond{}, s));
        // Iterate in chunks. A chunk's iterations past one whose recursive
        // residual met rtol do nothing (the true residual is the chunk's last
        // kernel), so what is left is counted by the iterations that ran; each
        // chunk runs at least one, and once done every later kernel returns at
        // once.
        const int chunk = 4;
        for (int chunks = 0;; chunks++) {
            PCG_CK(cudaMemcpyAsync(h->ctl_host, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
            PCG_CK(cudaStreamSynchronize(s));
            if (h->profile) prof_collect(h);
            const int left = maxit - h->ctl_host->iter;
            if (h->ctl_host->done || left <= 0 || chunks > maxit) break;
            const int todo = std::min(chunk, left);
            for (int k = 0; k < todo; k++) PCG_TRY(launch_iteration(h, k == 0, k + 1 == todo, Cond{}, s));
        }
    }
    Ctl &c = *h->ctl_host;
    if (c.done == 1 && c.bnorm == 0.0) k_zero<<<grid_rows(n), kBlock, 0, s>>>(h->x, n);
    PCG_LAUNCH_CK();
    PCG_CK(cudaMemcpyAsync(x, h->x, sizeof(double) * n, xdev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    if (res_hist) PCG_CK(cudaMemcpyAsync(res_hist, h->hist, sizeof(double) * (c.iter + 1), cudaMemcpyDefault, s));
    PCG_CK(cudaStreamSynchronize(s));
    if (iters) *iters = c.iter;
    h->last_true_rel = c.true_rel;
    int st = c.done ? c.status : AMG_ERR_NOCONV;
    if (st == AMG_ERR_NOCONV) set_error("pcg_solve: no convergence in %d iterations (rel %.3e)", maxit, c.rel);
    else if (st == AMG_ERR_BREAKDOWN) set_error("pcg_solve: breakdown (r.z <= 0 or p.Ap <= 0) at iteration %d", c.iter);
    else if (st == AMG_ERR_NAN) set_error("pcg_solve: NaN/Inf at iteration %d", c.iter);
    return st;
}

}  // namespace pcgamg

// Sums of doubles over a warp and a block on the integer pipe, shared by the
// solve kernels.
//
// On GB300 one float64 instruction of a warp holds its scheduler's float64
// pipe for 64 clocks whatever its active lanes (a dependent chain of adds ran
// 64.8 clocks per add; a quotient 563), so a shuffle tree of five adds costs
// 320 clocks of it in every warp, and the trees of the warps that share a
// scheduler queue up. Here a warp aligns its values to their largest exponent
// as 57-bit integers and adds those with the warp-wide integer reductions.
// The result does not depend on the order of the lanes; each value is rounded
// once at 2^-4 of the largest value's last place, so the sum is within
// 2 u max|x| + u |sum| of exact (u = 2^-53), where a tree of five float64 adds
// is within 5 u sum|x|.
#pragma once

#include <cstdint>

namespace pcgamg {

// Sum of x over the warp's lanes, in every lane. A NaN or an infinity gives
// NaN (the callers treat both alike).
__device__ __forceinline__ double warp_sum(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned ex = (hi >> 20) & 0x7ffu;
    const unsigned E = __reduce_max_sync(0xffffffffu, ex);
    if (E == 0x7ffu) return __longlong_as_double(0x7ff8000000000000ll);
    // |x| = m 2^(max(ex, 1) - 1075), q = |x| in units of 2^(max(E, 1) - 1079):
    // below 2^57, so 32 of them stay below 2^62
    const unsigned d = max(E, 1u) - max(ex, 1u);
    unsigned long long q = ((unsigned long long)((hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32 | lo) << 4;
    if (d) q = d < 59 ? (q + (1ull << (d - 1))) >> d : 0ull;
    const long long sq = hi >> 31 ? -(long long)q : (long long)q;
    // 26 + 26 + the signed rest: each field's sum over 32 lanes fits 32 bits
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)sq & 0x3ffffffu);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(sq >> 26) & 0x3ffffffu);
    const int s2 = __reduce_add_sync(0xffffffffu, (int)(sq >> 52));
    const long long t = ((long long)s2 << 52) + ((long long)s1 << 26) + (long long)s0;
    if (t == 0) return 0.0;
    const double f = __ll2double_rn(t);
    const int k = (int)max(E, 1u) - 1079, et = ((__double2hiint(f) >> 20) & 0x7ff) + k;
    return et > 0 && et < 0x7ff ? __hiloint2double(__double2hiint(f) + k * (1 << 20), __double2loint(f)) : scalbn(f, k);
}

// Block-wide sums of NV doubles per thread, in every lane of the block's first
// warp (blockDim a multiple of 32, at most 1024); only the first `warps` warps
// hold values, the others' count as zeros.
template <int NV>
__device__ __forceinline__ void block_sum(double (&a)[NV], int warps) {
    __shared__ double sh[NV][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < warps) {
#pragma unroll
        for (int v = 0; v < NV; v++) a[v] = warp_sum(a[v]);
        if (lane == 0) {
#pragma unroll
            for (int v = 0; v < NV; v++) sh[v][w] = a[v];
        }
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int v = 0; v < NV; v++) a[v] = warp_sum(lane < warps ? sh[v][lane] : 0.0);
    }
}

// This block's partial sums, slot v at partials[v gridDim.x + block].
template <int NV>
__device__ __forceinline__ void write_partials(double (&a)[NV], double *partials) {
    block_sum<NV>(a, blockDim.x >> 5);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int v = 0; v < NV; v++) partials[v * gridDim.x + blockIdx.x] = a[v];
    }
}

// Sums of the g partials of each slot, in the block's first warp. Every
// thread of the block takes part; a thread's own partials (blockDim apart) are
// added in order. In two steps, so that a caller can place other loads between
// them: the thread's first partials, then the sums.
template <int NV>
__device__ __forceinline__ void first_partials(const double *partials, int g, double (&a)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; v++) a[v] = (int)threadIdx.x < g ? __ldcg(partials + (int64_t)v * g + threadIdx.x) : 0.0;
}

template <int NV>
__device__ __forceinline__ void rest_partials(const double *partials, int g, double (&a)[NV]) {
    for (int k = threadIdx.x + blockDim.x; k < g; k += blockDim.x)
#pragma unroll
        for (int v = 0; v < NV; v++) a[v] += __ldcg(partials + (int64_t)v * g + k);
    block_sum<NV>(a, min((int)(blockDim.x >> 5), (g + 31) >> 5));
}

template <int NV>
__device__ __forceinline__ void sum_partials(const double *partials, int g, double (&a)[NV]) {
    first_partials<NV>(partials, g, a);
    rest_partials<NV>(partials, g, a);
}

}  // namespace pcgamg

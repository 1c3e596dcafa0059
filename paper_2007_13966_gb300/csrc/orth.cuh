// Device parts of the CGS2 orthogonalisation shared by the single and the batched FGMRES.
#pragma once

#include "common.cuh"

namespace ras {

// Block sums of acc[0 .. k) and, if self, of acc[KM], in a fixed order, into row v (k for
// the last) of `partials` (leading dimension ld) at column `at`; RED_THREADS threads.
// Eight rows at a time go through shared memory, where a warp adds 8 values per lane before
// its tree of shuffles: 13 warp-wide additions per row and warp, where a tree per warp and
// row takes 40, and FP64 runs at 2 per cycle and SM (9 rows of 608 blocks: 12 us of the
// 34 us that the dot products of one million cells took).
template <int KM>
__device__ __forceinline__ void block_rows(const double (&acc)[KM + 1], int k, int self, double *partials,
                                           long long ld, long long at) {
    __shared__ double sh[8][RED_THREADS];
    static_assert(RED_THREADS == 256, "a warp per row of eight");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int g = 0; g <= KM; g += 8) {
        if (g >= k && !(self && KM < g + 8)) continue;
        __syncthreads();
#pragma unroll
        for (int v = 0; v < 8; ++v)
            if (g + v <= KM) sh[v][threadIdx.x] = acc[g + v <= KM ? g + v : 0];
        __syncthreads();
        const int row = g + w;
        if (row < k || (self && row == KM)) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < RED_THREADS / 32; ++q) s += sh[w][lane + 32 * q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) partials[(row == KM ? k : row) * ld + at] = s;
        }
    }
}

// One cell of the first update and the second dot products in one pass over V:
// w -= sum_v h[v] V[v], then acc[v] += V[v] w (each value of V read once)
template <int KM>
__device__ __forceinline__ double update_dot(const double *V, long long ldv, long long i, int k, const double *h,
                                             double w, double (&acc)[KM + 1]) {
    double x[KM];
#pragma unroll
    for (int v = 0; v < KM; ++v) x[v] = v < k ? V[v * ldv + i] : 0.0;
#pragma unroll
    for (int v = 0; v < KM; ++v)
        if (v < k) w = fma(-h[v], x[v], w);
#pragma unroll
    for (int v = 0; v < KM; ++v)
        if (v < k) acc[v] = fma(x[v], w, acc[v]);
    return w;
}

}  // namespace ras

// Block-wide fp64 sums.
#pragma once

#include <cuda_runtime.h>

namespace fftlb {

// The sum over the block's NT threads into *out: whole warps, or one part of a
// warp (16 threads: fp64 columns of 16), whose shuffles name its own lanes alone.
template <int NT> __device__ __forceinline__ void block_sum_store(double v, double *out) {
    static_assert(NT % 32 == 0 || NT == 16 || NT == 8, "whole warps, or a power of two of lanes");
    constexpr int nl = NT < 32 ? NT : 32, nw = (NT + 31) / 32;
    constexpr unsigned lanes = nl == 32 ? 0xffffffffu : (1u << nl) - 1u;
    __shared__ double red[nw];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int w = nl / 2; w > 0; w >>= 1) v += __shfl_down_sync(lanes, v, w);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int i = 0; i < nw; ++i) s += red[i];
        *out = s;
    }
}

// The sums (the maximum for q == MAXQ) over the block's NT threads of NQ values
// each, handed to put(q, total) by one thread per value.  Through shared memory,
// a warp per value: shuffles by every warp over every value are five adds a
// thread and value on a pipe of two lanes a clock (k_inv_sites at 1024^2: 8 us of
// its 50).
template <int NQ, int NT, int MAXQ, typename Put>
__device__ __forceinline__ void block_totals(const double (&v)[NQ], double (&buf)[NQ][NT], const Put &put) {
    static_assert(NQ <= NT / 32, "a warp per value");
    const int tid = (int)threadIdx.x, q = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int i = 0; i < NQ; ++i) buf[i][tid] = v[i];
    __syncthreads();
    if (q >= NQ) return;
    double s = buf[q][lane];
#pragma unroll
    for (int j = 1; j < NT / 32; ++j) s = q == MAXQ ? fmax(s, buf[q][lane + 32 * j]) : s + buf[q][lane + 32 * j];
    for (int w = 16; w > 0; w >>= 1) {
        const double o = __shfl_down_sync(0xffffffffu, s, w);
        s = q == MAXQ ? fmax(s, o) : s + o;
    }
    if (lane == 0) put(q, s);
}

}  // namespace fftlb

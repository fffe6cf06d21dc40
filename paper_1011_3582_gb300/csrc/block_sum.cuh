// Sum of one fp64 value per thread over the block, stored by thread 0.
#pragma once

#include <cuda_runtime.h>

namespace fftlb {

__device__ __forceinline__ void block_sum_store(double v, double *out) {
    __shared__ double red[32];
    const int nw = (int)((blockDim.x + 31) >> 5), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int i = 0; i < nw; ++i) s += red[i];
        *out = s;
    }
}

}  // namespace fftlb

// The column kernels of kernels_col.cuh as the engine sees them.
#pragma once

#include <stddef.h>

#include "fft_types.h"

namespace fftlb {

// Threads per column of NY = E P values (0: no configuration, or a column
// per thread)
__host__ __device__ constexpr int col_p(int size, int NY) {
    return NY == 2048 || NY == 1536 ? 64
         : NY == 1024 || NY == 768 ? 32
         : NY == 512 ? (size == 8 ? 32 : 16)
         : NY == 384 || NY == 256 ? 16
         : NY == 192 || NY == 128 || NY == 96 || NY == 64 ? 8
         : NY == 48 || NY == 32 || NY == 24 || NY == 16 ? 4 : 0;
}
// stage 2 with two threads per P-point DFT (64 points do not fit one thread's
// registers; nor, in fp64 at two blocks per SM, do 32 of 512)
__host__ __device__ constexpr bool col_pair(int size, int NY) {
    return NY == 2048 || NY == 1536 || (NY == 512 && size == 8);
}
// columns per tile: 64 bytes of every row, 32 where a tile of 64 would leave
// one block per SM
__host__ __device__ constexpr int col_tw(int size, int NY) {
    return size == 4 ? (NY >= 1536 ? 4 : 8) : 4;
}

// one group of a launch: slots and multiplier
template <typename real> struct ColGroup {
    int in, out, add;   // add < 0: no addend
    real c0, c1, c3;
};

constexpr int kMaxColJobs = 40;   // groups of one launch

template <typename real> struct ColArgs {
    using C = typename cplx_of<real>::type;
    C *spec;
    const real *kx, *ky;
    const C *tw, *twt, *wp;   // [k1][l], [l][k1], exp(-2 pi i k / P)
    real scale;
    int h, ngroups;
    ColGroup<real> g[kMaxColJobs];
};

struct ColSet {
    const void *k = nullptr;
    int nt = 0, tw = 0;   // tw = 0: a column per thread
    size_t smem = 0;
};

// the kernel for columns of NY values (k == nullptr: none)
ColSet col_set_f32(int NY);
ColSet col_set_f64(int NY);

}  // namespace fftlb

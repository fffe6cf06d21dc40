// The column kernels of kernels_col.cuh as the engine sees them.
#pragma once

#include <stddef.h>

#include "fft_types.h"

namespace fftlb {

// Threads per column of NY = E P values (0: no configuration, or a column
// per thread).  fp64 at 24, 32 and 48: 8, so that the 4 columns of a tile fill a
// warp, which takes as long half empty; with 4 threads a column the two launches
// took 22.5 and 22.0 us on 96x48 (16.3, 15.6 so), 131 and 22.5 on 1024x48 (82,
// 16.2), 43 and 14.6 on 512x32 (37, 13.7), 39.5 and 14.5 on 512x24 (35.4, 13.1).
__host__ __device__ constexpr int col_p(int size, int NY) {
    return NY == 2048 || NY == 1536 ? 64
         : NY == 1024 || NY == 768 || NY == 512 ? 32
         : NY == 384 || NY == 256 ? 16
         : NY == 192 || NY == 128 || NY == 96 || NY == 64 || (size == 8 && (NY == 48 || NY == 32 || NY == 24)) ? 8
         : NY == 48 || NY == 32 || NY == 24 || NY == 16 ? 4 : 0;
}
// stage 2 with two threads per P-point DFT: 64 points do not fit one thread's
// registers; nor, in fp64 at two blocks per SM, do 32 of 512; and 16 values a
// thread instead of 32 leave the fp32 columns of 512 24 warps an SM instead of
// 16 (2048x512: convection 74 -> 69.5 us)
__host__ __device__ constexpr bool col_pair(int size, int NY) { return NY == 2048 || NY == 1536 || NY == 512; }
// columns per tile: 64 bytes of every row, 32 where a tile of 64 would leave
// one block per SM
__host__ __device__ constexpr int col_tw(int size, int NY) {
    return size == 4 ? (NY >= 1536 ? 4 : 8) : 4;
}
// tables in shared memory (see kernels_col.cuh)
__host__ __device__ constexpr bool col_tables(size_t size, int NY) { return size == 4 && NY < 1536; }

// one group of a launch: input slot (or distribution), output slot and
// multiplier with the inverse normalisation folded in
template <typename real> struct ColGroup {
    int in, out, from_f;
    real c0, c1, c3;
};

// The tables of kcol_reg as one block: stage-1 twiddles exp(-2 pi i l k1 / NY) in
// the orders [k1][l] and [l][k1], exp(-2 pi i k / P) (k < P), k_y of the NY bins
template <typename real> __host__ __device__ constexpr unsigned col_table_bytes(int NY, int P) {
    return (unsigned)((2 * NY + P) * 2 * sizeof(real) + NY * sizeof(real));
}

constexpr int kMaxColJobs = 40;   // groups of one launch

// the gradient of caller fields (dx_row, dy_col): row and column tables
template <typename real> struct GradArgs {
    using C = typename cplx_of<real>::type;
    const double2 *g;   // [fields][ny][nx / 2] pairs of fp64 values
    double2 *out;       // [2 fields][ny][nx / 2]
    const C *rtab, *ctab;
    const real *ky;
    int h, ny, nrows;   // nrows = fields ny
    int *err;
};

// the gradient energy of a real field rho [ny][nx]
template <typename real> struct EnergyArgs {
    using C = typename cplx_of<real>::type;
    const C *rho;
    const C *rtab, *ctab;
    const real *ky;
    double *partial_x, *partial_y;   // one value per block of energy_row / energy_col
    int h, ny;
    int *err;
};

template <typename real> struct ColArgs {
    using C = typename cplx_of<real>::type;
    C *spec;
    const C *f;               // the stage state [run][33][ny][nx], as rows of nx / 2 complex values
    const real *kx, *ky;
    const C *tab;             // table block, see col_table_bytes
    int *err;
    int h, ngroups;
    ColGroup<real> g[kMaxColJobs];
};

struct ColSet {
    const void *k = nullptr, *dy = nullptr, *energy = nullptr;
    int nt = 0, tw = 0;   // tw = 0: a column per thread
    size_t smem = 0;
};

// the kernel for columns of NY values (k == nullptr: none)
ColSet col_set_f32(int NY);
ColSet col_set_f64(int NY);

}  // namespace fftlb

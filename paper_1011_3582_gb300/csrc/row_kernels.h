// The row and column kernels of kernels_row.cuh / kernels_col.cuh as the
// engine sees them: configurations, arguments and launch records.  The
// kernels are instantiated in rows_*.cu and cols_*.cu, one set of lengths and
// one precision each, so that they compile in parallel; they take the
// velocity set and every constant as arguments and keep no state.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <vector_types.h>

#include "fft_types.h"

namespace fftlb {

// Lanes per row of a half row of H = E P complex values (0: no
// configuration).  E points of the first stage sit in each lane's registers:
// up to 32 (fp32) or 24 (fp64) complex values.
__host__ __device__ constexpr int row_p(int H) {
    return H == 1024 || H == 768 || H == 512 ? 32
         : H == 384 || H == 256 ? 16
         : H == 192 || H == 128 || H == 96 || H == 64 ? 8
         : H == 48 || H == 32 || H == 24 || H == 16 ? 4 : 0;
}
// threads per block
__host__ __device__ constexpr int row_nt(int, int H) { return row_p(H) == 32 ? 256 : 128; }
// blocks per row (cluster size): as many as give every row group one
// distribution row, at most 4
__host__ __device__ constexpr int row_cs(int, int H) { return row_p(H) >= 16 ? 4 : row_p(H) == 8 ? 2 : 1; }
// complex values between rows in shared memory: rows of one memory phase
// (half a warp of 8-byte, a quarter of 16-byte values) in different banks
__host__ __device__ constexpr int row_stride(int size, int H) {
    return H + (row_p(H) * 2 * size < 128 && row_p(H) < 16 ? row_p(H) : 0);
}

template <typename real> struct RowArgs {
    using C = typename cplx_of<real>::type;
    int ny, nrun;
    real dt, itau, a, b, K, H, q, zeta, scale_x, alpha, beta;
    const real *f;      // K1: the stage state [run][33][ny][nx]
    real *fields, *aux;
    C *spec;
    const real *fcur, *fbase;   // K5
    real *fout;
    const C *tw, *wp, *wh;      // stage-1 twiddles; exp(-2 pi i k / nx), k <= H / 2, and half of it
    const real *kx;
    int *err;
    real vx[33], vy[33], v2[33];
    real Fk[4][4], Fkl[4][4];   // Eq. 4's polynomials (fp32: hi and lo parts)
};

struct RowSet {
    const void *k1 = nullptr, *k3 = nullptr, *k5 = nullptr;
    int nt = 0, cs = 1;
    size_t smem1 = 0, smem3 = 0, smem5 = 0;
};

// the kernels for half rows of H values (k1 == nullptr: none)
RowSet row_set_f32_p2(int H);
RowSet row_set_f32_r3(int H);
RowSet row_set_f64_p2(int H);
RowSet row_set_f64_r3(int H);

}  // namespace fftlb

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
__host__ __device__ constexpr int row_p(int size, int H) {
    return H == 1024 || H == 768 || H == 512 ? 32
         : H == 384 || H == 256 ? 16
         : H == 192 || H == 128 || H == 96 || H == 64 || (size == 8 && (H == 48 || H == 32)) ? 8
         : H == 48 || H == 32 || H == 24 || H == 16 ? 4 : 0;
}
// threads per block
__host__ __device__ constexpr int row_nt(int size, int H) { return row_p(size, H) == 32 ? 256 : 128; }
// ... of K3, whose 11 derivative rows fill half the row groups: more, smaller
// blocks keep the warps busy (2048^2 fp32 272 -> 183 us, 384^2 25 -> 19, 1024^2
// fp64 889 -> 749; shorter fp64 rows lose by it: 256^2 95 -> 104)
__host__ __device__ constexpr int row_nt3(int size, int H) { return size == 4 && row_p(size, H) < 32 ? 64 : 128; }
// blocks per row (cluster size): as many as give every row group one
// distribution row, at most 4
__host__ __device__ constexpr int row_cs(int size, int H) { return row_p(size, H) >= 16 ? 4 : row_p(size, H) == 8 ? 2 : 1; }
// complex values between rows in shared memory: rows of one memory phase
// (half a warp of 8-byte, a quarter of 16-byte values) in different banks
__host__ __device__ constexpr int row_stride(int size, int H) {
    return H + (row_p(size, H) * 2 * size < 128 && row_p(size, H) < 16 ? row_p(size, H) : 0);
}

// The tables of the row kernels as one block of bytes: wh[k] = exp(-2 pi i k /
// 2H) / 2 (k < H / 2), kx[k] (k < H), the stage-1 twiddles tw[k1 P + l] = exp(-2
// pi i l k1 / H), wp[k] = exp(-2 pi i k / 2H) (k < H / 2); offsets of its parts,
// each a multiple of 16 bytes
template <typename real> struct RowTable {
    static __host__ __device__ constexpr unsigned up(unsigned b) { return (b + 15u) & ~15u; }
    static __host__ __device__ constexpr unsigned half(int H) { return up(H / 2 * 2 * sizeof(real)); }
    static __host__ __device__ constexpr unsigned kx(int H) { return half(H); }
    static __host__ __device__ constexpr unsigned tw(int H) { return kx(H) + up(H * sizeof(real)); }
    static __host__ __device__ constexpr unsigned wp(int H) { return tw(H) + H * 2 * sizeof(real); }
    static __host__ __device__ constexpr unsigned bytes(int H) { return wp(H) + half(H); }
};

template <typename real> struct RowArgs {
    using C = typename cplx_of<real>::type;
    int ny, nrun;
    real dt, itau, a, b, K, H, q, zeta, scale_x, alpha, beta;
    const real *f;      // K1: the stage state [run][33][ny][nx]
    C *spec;            // the slots [run][NSLOT][ny][nx / 2]
    const real *fcur, *fbase;   // K5
    real *fout;
    const C *tab;               // table block, see RowTable
    int *err;
    real vx[33], vy[33], v2[33];
    real Fk[4][4], Fkl[4][4];   // Eq. 4's polynomials (fp32: hi and lo parts)
};

struct RowSet {
    const void *k1 = nullptr, *k3 = nullptr, *k5 = nullptr;
    const void *dx = nullptr, *energy = nullptr;   // single-row kernels: ng rows a block, smem_rows bytes
    int ng = 1;
    size_t smem_rows = 0;
    int nt = 0, nt3 = 0, cs = 1;
    size_t smem1 = 0, smem3 = 0, smem5 = 0;
};

// the kernels for half rows of H values (k1 == nullptr: none)
RowSet row_set_f32_p2(int H);
RowSet row_set_f32_r3(int H);
RowSet row_set_f64_p2(int H);
RowSet row_set_f64_r3(int H);

}  // namespace fftlb

// What the kernels of one stage share with the engine: the spectrum slots,
// the derivative rows and the column-pass groups.
#pragma once

namespace fftlb {

constexpr int Q = 33;
constexpr int NMOV = 32;

// The windowed derivative multipliers are separable: D_x = i k_x (a function
// of k_x alone), D_y = i k_y, and the second derivatives are their products
// (Eqs. K1-K4 with the real part taken after each derivative, so that the
// Nyquist bins carry zero).  So a derivative along one axis needs transforms
// along that axis alone:
//   - i k_x terms are pointwise products in the row spectrum: i k_x X / nx (the
//     1 / nx completes the unnormalised inverse row transform);
//   - i k_y terms are column passes (forward, multiplier, inverse) of real
//     fields as they are: two neighbouring real columns packed as one complex
//     column x = f(2m) + i f(2m+1) take the multiplier together, because D_y maps
//     real columns to real columns.  A row of nx reals and a row spectrum of
//     nx / 2 complex values share one layout, so the column kernels do not
//     distinguish them.
// Convection (v_x D_x + v_y D_y) f_i: the 8 velocities with v_y = 0 take
// i v_x k_x f^ / nx in K1 and no column pass; the 8 with v_x = 0 take a column
// pass of f_i itself and no row transform; the other 16 take both.  Level 1:
// D_y of rho, T, Pi, g and D_yy of rho, u_y are column passes of the real
// fields; only D_y u_x and D_y u_y, which also enter mixed derivatives, start
// from row spectra.  Level 2: D_x of Lambda_xx, Lambda_xy, Phi_x is a
// forward row in K3 and an inverse row in K3 (which then adds it to the
// numerators in SLOT_A) or, for the k*_row kernels, in K5 (from SLOT_X); the
// column pass takes the real Lambda_xy, Lambda_yy, Phi_y in place.
// A stage has 71 row transforms (30 in K1, 17 in K3, 24 in K5) and 35 column
// passes; with every derivative through the row spectrum it was 93 (38, 20,
// 35) and as many column passes.
//
// slots: [ny][nx / 2] complex values or [ny][nx] reals
constexpr int SLOT_RHO = 32, SLOT_UX = 33, SLOT_UY = 34, SLOT_T = 35, SLOT_PI = 36, SLOT_G = 37;   // row spectra
constexpr int SLOT_D1 = 38;      // column-pass outputs of level 1, see D1_* below
enum { D1_UXY, D1_UYY, D1_RY, D1_RYY, D1_TY, D1_PIY, D1_GY, D1_UYYY, ND1 };   // the first two are row spectra
constexpr int SLOT_L2 = SLOT_D1 + ND1;   // Lambda_xy, Lambda_yy, Phi_y, then their D_y (real)
constexpr int SLOT_F = SLOT_L2 + 3;      // rho, u_x, u_y, T, Pi, g (real)
constexpr int SLOT_A = SLOT_F + 6;       // numerators of C + C_q, B_x, B_y (real)
constexpr int SLOT_X = SLOT_A + 3;       // k*_row: row spectra of the d_x of Phi_x, Lambda_xx, Lambda_xy
constexpr int NSLOT = SLOT_X + 3;

// K3's rows: the first NSP are inverse-transformed (those without a source
// slot are formed from the others: lap rho's k_x part from rho^, d_x div u from
// u_x^ and D_y u_y, the k_x part of d_y div u from D_y u_x), the rest are real
enum { D_RX, D_LAP, D_UXX, D_UXY, D_UYX, D_UYY, D_DIVX, D_DIVY, D_TX, D_PIX, D_GX, NSP,
       D_RY = NSP, D_RYY, D_TY, D_PIY, D_GY, D_UYYY, D_RHO, D_T, NK3 };
__host__ __device__ constexpr int k3_src_slot(int o) {
    return o == D_RX ? SLOT_RHO : o == D_UXX ? SLOT_UX : o == D_UYX ? SLOT_UY : o == D_TX ? SLOT_T
         : o == D_PIX ? SLOT_PI : o == D_GX ? SLOT_G : o == D_UXY ? SLOT_D1 + D1_UXY : o == D_UYY ? SLOT_D1 + D1_UYY
         : o == D_RY ? SLOT_D1 + D1_RY : o == D_RYY ? SLOT_D1 + D1_RYY : o == D_TY ? SLOT_D1 + D1_TY
         : o == D_PIY ? SLOT_D1 + D1_PIY : o == D_GY ? SLOT_D1 + D1_GY : o == D_UYYY ? SLOT_D1 + D1_UYYY
         : o == D_RHO ? SLOT_F : o == D_T ? SLOT_F + 3 : -1;
}

// The 6 directions of a ring (Eq. 1) whose convection term takes row
// transforms: 0, 1, 3, 4, 5, 7 (v_x != 0)
__host__ __device__ constexpr int ring_dir(int t) { return t < 2 ? t : t < 5 ? t + 1 : 7; }
__host__ __device__ constexpr int ring_pos(int r) { return r < 2 ? r : r < 6 ? r - 1 : 5; }   // its inverse

// One column-pass group: up to 2 outputs of one input, each M(kx, ky) * input
// with M = i (c0 k_x + c1 k_y) + (c2 k_x^2 + c3 k_y^2 + c4 k_x k_y).  The stage's
// groups have one output, take slot in_slot, or distribution in_slot of the
// stage state where from_f is set, and multiply by scale: 1 / (nx ny) for row
// spectra, 1 / ny for real fields.
struct GroupDesc {
    int nin, nout;
    int in_slot[2];
    int out_slot[6];
    int nterm[6];
    int term_in[6][2];
    double c[6][2][5];
    int from_f;
    double scale;
};

}  // namespace fftlb

// What the kernels of one stage share with the engine: the spectrum slots,
// the derivative rows and the column-pass groups.
#pragma once

namespace fftlb {

constexpr int Q = 33;
constexpr int NMOV = 32;

// spectrum slots
constexpr int SLOT_RHO = 32, SLOT_UX = 33, SLOT_UY = 34, SLOT_T = 35, SLOT_PI = 36, SLOT_G = 37;
constexpr int SLOT_D1 = 38;      // 15 level-1 derivative outputs
constexpr int ND1 = 15;
constexpr int SLOT_L2 = 53;      // Lxx, Lxy, Lyy, Phx, Phy; outputs in 53, 55, 56
constexpr int NSLOT = 58;
enum { D_RX, D_RY, D_LAP, D_UXX, D_UXY, D_UYX, D_UYY, D_DIVX, D_DIVY, D_TX, D_TY, D_PIX, D_PIY, D_GX, D_GY };

// The windowed derivative multipliers are separable: D_x = i k_x (a
// function of k_x alone), D_y = i k_y, and the second derivatives are their
// products (Eqs. K1-K4 with the real part taken after each derivative, so
// that the Nyquist bins carry zero).  A derivative whose multiplier depends
// on k_x alone needs no column transform: in the row-transformed slot it is
// the pointwise product i k_x X / nx (the 1 / nx that the column pass would
// leave).  So the column pass forms only derivatives in k_y alone, each of
// one input: d_y of rho, u_x, u_y, T, Pi, g and d_yy of rho, u_y; and the
// row kernel K3 forms the rest from the row spectra of rho, u_x, u_y, T,
// Pi, g and of those before its inverse rows:
//   rho_x = i k_x rho^ / nx, lap rho = d_yy rho - k_x^2 rho^ / nx,
//   u_xx = i k_x u_x^ / nx, u_yx = i k_x u_y^ / nx,
//   d_x(div u) = i k_x (u_xx + u_yy), d_y(div u) = d_yy u_y + i k_x (d_y u_x),
//   T_x, Pi_x, g_x = i k_x (.)^ / nx.
// With one input and one output each, the level-1 passes are 8 more groups
// of the convection launch.  A launch of their own for rho (two outputs) and
// u (two inputs, two outputs) transformed two inputs fewer, but with three
// tiles and 219 KB a block it left most SMs with one job's latency: 22.5 us
// at 1024^2 in fp32, against the 9 us these jobs add to the convection
// launch (69.8 -> 78.7 us); 48 and 15.9 us against none on 64^2 fp64 and fp32.
// Level 2 in the same way: d_x Lambda_xx + d_y Lambda_xy is the column
// pass of d_y Lambda_xy plus i k_x Lambda_xx^ / nx, formed by K3 (add_slot).
// k3_src_slot(o): the slot K3 loads into its row o (-1: formed in K3).
__host__ __device__ constexpr int k3_src_slot(int o) {
    return o == D_RX ? SLOT_RHO : o == D_UXX ? SLOT_UX : o == D_UYX ? SLOT_UY : o == D_TX ? SLOT_T
         : o == D_PIX ? SLOT_PI : o == D_GX ? SLOT_G : o == D_DIVX ? -1 : SLOT_D1 + o;
}
// K3's level-2 outputs: row r of Lambda_xx, Lambda_xy, Lambda_yy, Phi_x,
// Phi_y goes to slot k3_raw_slot(r) as it is and to slot k3_mul_slot(r)
// times i k_x / nx (-1: not written)
__host__ __device__ constexpr int k3_raw_slot(int r) {
    return r == 1 ? SLOT_L2 + 1 : r == 2 ? SLOT_L2 + 2 : r == 4 ? SLOT_L2 + 4 : -1;
}
__host__ __device__ constexpr int k3_mul_slot(int r) {
    return r == 0 ? SLOT_L2 + 0 : r == 1 ? SLOT_D1 + D_DIVX : r == 3 ? SLOT_L2 + 3 : -1;
}

// One column-pass group: up to 2 input spectra and 6 outputs; every output
// is a sum of up to 2 terms M(kx, ky) * input, with
// M = i (c0 k_x + c1 k_y) + (c2 k_x^2 + c3 k_y^2 + c4 k_x k_y).
// add_slot >= 0 (groups of one input and one output, the convection kernels
// only): the column inverse of that output is added to slot add_slot's
// values at the same positions (a term that needs no column transform,
// formed by the row kernel that wrote add_slot).
struct GroupDesc {
    int nin, nout;
    int in_slot[2];
    int out_slot[6];
    int nterm[6];
    int term_in[6][2];
    double c[6][2][5];
    int add_slot;
};

}  // namespace fftlb

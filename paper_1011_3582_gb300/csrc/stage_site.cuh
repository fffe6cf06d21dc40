// Pointwise arithmetic of a stage shared by the kernel families.
#pragma once

#include "stage_layout.cuh"

namespace fftlb {

// Level 2 at one site from K3's rows (d(o) = row o): Lambda (Eq. 19), Phi =
// 2 q rho T grad T (Eq. 23) and the numerators of C (Eq. 22) and B (Eq. 21)
// without the divergences of Lambda and Phi.
template <typename real> struct Level2 {
    real Lxx, Lxy, Lyy, Phx, Phy, Cn, Bx, By;
};
template <typename real, typename Row, typename Par>
__device__ __forceinline__ Level2<real> level2_site(const Row &d, const Par &P) {
    const real rho = d(D_RHO), T = d(D_T);
    const real rx = d(D_RX), ry = d(D_RY), lap = d(D_LAP) + d(D_RYY);
    const real uxx = d(D_UXX), uxy = d(D_UXY), uyx = d(D_UYX), uyy = d(D_UYY);
    const real divx = d(D_DIVX), divy = d(D_DIVY) + d(D_UYYY);
    const real M = P.K + P.H * T;
    const real Pi = rho * T / (real(1) - P.b * rho) - P.a * rho * rho - rho * T;
    const real grad2 = rx * rx + ry * ry;
    const real iso = -(rho * T * (rx * d(D_GX) + ry * d(D_GY))) - M * (rho * lap + real(0.5) * grad2);   // Eq. 19
    Level2<real> o;
    o.Lxx = M * rx * rx + iso;
    o.Lxy = M * rx * ry;
    o.Lyy = M * ry * ry + iso;
    const real div = uxx + uyy;
    const real Ldu = o.Lxx * uxx + o.Lxy * (uyx + uxy) + o.Lyy * uyy;
    o.Cn = Pi * div + Ldu - P.zeta * div * div + P.a * rho * rho * div +
           P.K * (real(-0.5) * grad2 * div - rho * (rx * divx + ry * divy) -
                  (rx * (uxx * rx + uyx * ry) + ry * (uxy * rx + uyy * ry)));   // Eq. 22
    o.Bx = d(D_PIX) - P.zeta * divx;   // Eq. 21 without d_b Lambda_ab
    o.By = d(D_PIY) - P.zeta * divy;
    const real q2 = real(2) * P.q * rho * T;   // Eq. 23
    o.Phx = q2 * d(D_TX);
    o.Phy = q2 * d(D_TY);
    return o;
}

// One value's Runge-Kutta combination: f + dt rhs, or with a base state fb
// (1 - beta) fb + beta (f + dt rhs) as fb + beta ((f - fb) + dt rhs).  In fp32
// the weights 1/3 and 2/3 rounded add up to 1 + 3e-8, which scaled every f by
// that each step (a mass drift of 2e-8 a step); here f and fb, which are close,
// are subtracted without rounding and the small sum is rounded once.
template <typename real>
__device__ __forceinline__ real rk_combine(bool with_base, real beta, real dt, real f, real fb, real rhs) {
    return with_base ? fb + beta * ((f - fb) + dt * rhs) : f + dt * rhs;
}

}  // namespace fftlb

// In-register DFTs of the row and column configurations (kernels_wr.cuh,
// kernels_row.cuh) beyond those of fft_device.cuh: 32 points, and 3 M points
// (M = 2, 4, 8) as three M-point DFTs and one radix-3 step with the
// constants W_3M^k (decimation in time).
#pragma once

#include "fft_device.cuh"

namespace fftlb {

// cos(2 pi k / 24)
__host__ __device__ constexpr double cos24(int k) {
    k = ((k % 24) + 24) % 24;
    if (k > 12) k = 24 - k;
    const double s = k > 6 ? -1.0 : 1.0;
    if (k > 6) k = 12 - k;
    return s * (k == 0 ? 1.0
              : k == 1 ? 0.96592582628906828675
              : k == 2 ? 0.86602540378443864676
              : k == 3 ? 0.70710678118654752440
              : k == 4 ? 0.5
              : k == 5 ? 0.25881904510252076235
                       : 0.0);
}
__host__ __device__ constexpr double sin24(int k) { return cos24(k - 6); }

template <int M, int DIR, typename C> struct DFT3M {
    __device__ __forceinline__ static void run(C *v) {
        using R = decltype(v[0].x);
        C y[3][M];
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int r = 0; r < 3; ++r) y[r][m] = v[3 * m + r];
#pragma unroll
        for (int r = 0; r < 3; ++r) SmallDFT<M, DIR, C>::run(y[r]);
        constexpr int U = 24 / (3 * M);   // W_3M^k = W_24^(U k)
#pragma unroll
        for (int k = 0; k < M; ++k) {
            C t[3] = {y[0][k], y[1][k], y[2][k]};
            if (k > 0) {
                t[1] = mul_wc<DIR>(t[1], R(cos24(U * k)), R(sin24(U * k)));
                t[2] = mul_wc<DIR>(t[2], R(cos24(2 * U * k)), R(sin24(2 * U * k)));
            }
            SmallDFT<3, DIR, C>::run(t);
#pragma unroll
            for (int s = 0; s < 3; ++s) v[k + M * s] = t[s];
        }
    }
};
template <int DIR, typename C> struct SmallDFT<6, DIR, C> : DFT3M<2, DIR, C> {};
template <int DIR, typename C> struct SmallDFT<12, DIR, C> : DFT3M<4, DIR, C> {};
template <int DIR, typename C> struct SmallDFT<24, DIR, C> : DFT3M<8, DIR, C> {};

// cos(2 pi k / 32), k = 0..8 (the rest by symmetry)
__device__ __forceinline__ constexpr double cos32(int k) {
    return k == 0 ? 1.0
         : k == 1 ? 0.98078528040323044913
         : k == 2 ? 0.92387953251128675613
         : k == 3 ? 0.83146961230254523708
         : k == 4 ? 0.70710678118654752440
         : k == 5 ? 0.55557023301960222474
         : k == 6 ? 0.38268343236508977173
         : k == 7 ? 0.19509032201612826785
                  : 0.0;
}

// W_32^k = exp(DIR 2 pi i k / 32) for 0 <= k < 16, compile-time after unrolling
template <int DIR, typename R>
__device__ __forceinline__ void w32(int k, R &c, R &s) {
    const double cc = k <= 8 ? cos32(k) : -cos32(16 - k);
    const double ss = k <= 8 ? cos32(8 - k) : cos32(k - 8);
    c = R(cc);
    s = R(DIR < 0 ? -ss : ss);
}

// 32-point DFT as two 16-point DFTs of the even and odd inputs and one
// radix-2 step with the constants W_32^k
template <int DIR, typename C> struct SmallDFT<32, DIR, C> {
    __device__ __forceinline__ static void run(C *v) {
        using R = decltype(v[0].x);
        C e[16], o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            e[i] = v[2 * i];
            o[i] = v[2 * i + 1];
        }
        SmallDFT<16, DIR, C>::run(e);
        SmallDFT<16, DIR, C>::run(o);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            R c, s;
            w32<DIR, R>(k, c, s);
            if (sizeof(R) == 8 && k > 0 && k != 8) {
                butterfly(e[k], o[k], c, s);
                v[k] = e[k];
                v[k + 16] = o[k];
                continue;
            }
            const C t = k == 0 ? o[k] : C{o[k].x * c - o[k].y * s, o[k].x * s + o[k].y * c};
            v[k] = cadd(e[k], t);
            v[k + 16] = csub(e[k], t);
        }
    }
};

}  // namespace fftlb

// Column passes without staged tiles, in fp32 and fp64:
//   kcol_reg   lengths 16 .. 2048 = 2^p and 24 .. 1536 = 3 2^p: one job (a
//              tile of TW spectrum columns of one group) per block;
//   kcol_line  lengths 4, 6, 8, 12: one column per thread, in registers.
// Every group has one input (a slot or a distribution of the stage state) and
// one output (which may be the same slot): forward transform, multiplier
// i (c0 k_x + c1 k_y) or c3 k_y^2, inverse.
//
// A column of NY = E P values is transformed by P threads in two register
// stages: thread (c, l) takes the E-point DFT of x[l + P t], times W_NY^(l k1),
// and stores it transposed in shared memory; thread (c, k1) takes the P-point
// DFTs over l, applies the multiplier to X[k1 + E k2], and goes back the same
// way (P points by two threads, with one shuffle each way, where they do not
// fit one thread's registers).  The values come straight from global memory
// into registers, so the tile passes through shared memory twice, a block holds
// one tile, and several blocks on an SM overlap loads and transforms.  A
// persistent kernel that staged tiles by tensor copies (two buffers, L2
// prefetch) took 77.7 us for the convection launch of 1024^2 fp32 and 17.9 for
// level 2 (one job's latency), 24.5 and 11.8 at 512^2; this one 78 and 14.5,
// 22.5 and 8.2.  Both are held by the latency of shared memory and of the loads
// at 16 warps per SM (44% of the issue slots, 3.9 TB/s at 1024^2, 3.0 with the
// 32-byte rows of 2048); 24 warps, which 16 values a thread allow, gain 6% (see
// col_minb).
// The packed column 0 of the tile at k_x = 0 (DC real, row-Nyquist imaginary)
// needs no pairing of (k_y, -k_y): both columns it carries take the multiplier
// at k_x = 0, because the Nyquist bin of k_x is zero.
// The tables of the 8-wide fp32 tiles come by one bulk copy that overlaps the
// tile's loads: read through L1, they were cold in every launch, a latency per
// handful of twiddles (one job's time on 384^2: 13.8 us, 10.2 with the copy).
// 4-wide tiles are hardly larger than their tables (2048^2: convection 479 us
// with the copy, 372 through L1), and fp64's arithmetic hides the latency.
#pragma once

#include "async_copy.cuh"
#include "col_kernels.h"
#include "block_sum.cuh"
#include "fft_small.cuh"
#include "stage_layout.cuh"

namespace fftlb {

namespace ck {

template <typename real, int NY> struct Col {
    using C = typename cplx_of<real>::type;
    static constexpr int P = col_p(sizeof(real), NY), E = NY / P;
    static constexpr bool PAIR = col_pair(sizeof(real), NY);   // stage 2: two threads per P-point DFT
    static constexpr int PH = PAIR ? P / 2 : P;
    static constexpr int TW = col_tw(sizeof(real), NY), NT = TW * P;
    // rows of one memory phase (16 8-byte or 8 16-byte values) in different banks
    static constexpr bool TABS = col_tables(sizeof(real), NY);   // tables in shared memory
    static constexpr int PHASE = 128 / (int)sizeof(C), SW = TW < PHASE ? PHASE / TW - 1 : 0;
};

// a table value from shared or (read-only) global memory
template <bool SH, typename T> __device__ __forceinline__ T tab(const T *p) {
    if constexpr (SH) return *p;
    else return __ldg(p);
}

// position of stage-1 output (l, k1) of column c
template <typename real, int NY> __device__ __forceinline__ int cp(int c, int l, int k1) {
    using G = Col<real, NY>;
    return (k1 * G::P + (l ^ (k1 & G::SW))) * G::TW + c;
}

template <typename real, int NY> constexpr int col_minb() {
    using G = Col<real, NY>;
    // threads an SM: 255 registers for more than 16 fp64 complex values a
    // thread, 128 up to there and for 32 fp32 ones, 85 for 16 of those on columns
    // of 256 and 512 (2048x256: convection 34.7 us with 128, 30.6 with 85, 30.7
    // with 64; 2048x512: 74, 69.5, 75.7).  Shorter columns keep 128: with 85 those
    // of 128 spill (2048x128: 18.6 us with 128, 20.8 with 85; 1024x128 12.4, 14.4;
    // 16 runs of 128^2 309, 317 a step), 192, 96 and 64 take as long either way
    constexpr bool half = G::E <= 16 && G::PH <= 16;
    constexpr int nt = sizeof(real) == 4 ? (half && NY >= 256 ? 768 : 512) : half ? 512 : 256;
    return nt / G::NT > 16 ? 16 : nt / G::NT;
}

// The tables of kcol_reg's length in shared memory behind the tile (copied by
// thread 0 while the tile loads) or in global memory.
template <typename real, int NY> struct ColTab {
    using G = Col<real, NY>;
    using C = typename G::C;
    const C *tw, *twt, *wp;
    const real *ky;
    __device__ __forceinline__ ColTab(C *tile, const C *g) {
        tw = G::TABS ? tile + (size_t)NY * G::TW : g;
        twt = tw + NY;
        wp = twt + NY;
        ky = reinterpret_cast<const real *>(wp + G::P);
    }
    static __device__ __forceinline__ void issue(C *tile, const C *g, uint64_t *bar) {
        if (G::TABS && threadIdx.x == 0) {
            mbar_init(bar, 1);
            mbar_init_fence();
            mbar_expect_tx(bar, col_table_bytes<real>(NY, G::P));
            bulk_g2s(tile + (size_t)NY * G::TW, g, col_table_bytes<real>(NY, G::P), bar);
        }
    }
    // the block's wait; false if it ran out (the copy is no longer in flight)
    static __device__ __forceinline__ bool wait(uint64_t *bar, int *err) {
        if constexpr (G::TABS) {
            __syncthreads();   // the barrier is initialised before any thread polls it
            if (!block_wait(bar, 0, err)) {
                mbar_wait_bounded(bar, 0);
                return false;
            }
        }
        return true;
    }
};

// The passes of thread (c, jl) over a tile: v = x[jl + P t] of column c in; with
// INV, v = the inverse transform of mult(k, X[k]) out, otherwise mult sees
// every X[k] once and v is undefined.  Returns false if the tables never came.
template <typename real, int NY, bool INV, typename Mult>
__device__ __forceinline__ bool col_pass(typename Col<real, NY>::C (&v)[Col<real, NY>::E], typename Col<real, NY>::C *T,
                                         const ColTab<real, NY> &tb, uint64_t *bar, int *err, int c, int jl,
                                         const Mult &mult) {
    using G = Col<real, NY>;
    using C = typename G::C;
    constexpr int E = G::E, P = G::P, PH = G::PH, TW = G::TW;
    SmallDFT<E, -1, C>::run(v);
    if (!ColTab<real, NY>::wait(bar, err)) return false;
#pragma unroll
    for (int k1 = 1; k1 < E; ++k1) v[k1] = cmul(v[k1], tab<G::TABS>(tb.tw + k1 * P + jl));
#pragma unroll
    for (int k1 = 0; k1 < E; ++k1) T[cp<real, NY>(c, jl, k1)] = v[k1];
    __syncthreads();
    // stage 2: forward, multiplier, inverse, conjugate twiddles
    if constexpr (!G::PAIR) {
#pragma unroll
        for (int q = 0; q < (E + P - 1) / P; ++q) {
            const int k1 = jl + P * q;
            if (E % P == 0 || k1 < E) {
                C u[P];
#pragma unroll
                for (int l = 0; l < P; ++l) u[l] = T[cp<real, NY>(c, l, k1)];
                SmallDFT<P, -1, C>::run(u);
#pragma unroll
                for (int k2 = 0; k2 < P; ++k2) u[k2] = mult(k1 + E * k2, u[k2]);
                if constexpr (INV) {
                    SmallDFT<P, +1, C>::run(u);
#pragma unroll
                    for (int l = 0; l < P; ++l)
                        T[cp<real, NY>(c, l, k1)] = l == 0 ? u[l] : cmul(u[l], cconj(tab<G::TABS>(tb.twt + l * E + k1)));
                }
            }
        }
    } else if (jl < 2 * E) {   // (whole warps)
        // threads (k1, gg) = (jl / 2, jl % 2) hold the even (gg = 0) and the
        // odd l; X[k2' + PH s] = V0[k2'] + (-1)^s W_P^k2' V1[k2']: thread gg
        // takes k2' in [PH gg / 2, PH (gg + 1) / 2), exchanging the other
        // half with its neighbour, and the inverse goes the same way back
        constexpr int HH = PH / 2;
        const int k1 = jl >> 1, gg = jl & 1;
        C u[PH];
#pragma unroll
        for (int m = 0; m < PH; ++m) u[m] = T[cp<real, NY>(c, gg + 2 * m, k1)];
        SmallDFT<PH, -1, C>::run(u);
#pragma unroll
        for (int i = 0; i < HH; ++i) {
            const C send = gg ? u[i] : u[HH + i];
            C recv;
            recv.x = __shfl_xor_sync(0xffffffffu, send.x, TW);
            recv.y = __shfl_xor_sync(0xffffffffu, send.y, TW);
            const C a = gg ? recv : u[i], b = gg ? u[HH + i] : recv;
            const int k2 = HH * gg + i;
            const C w = tab<G::TABS>(tb.wp + k2);   // W_P^k2
            const C t = cmul(b, w);
            const C x0 = mult(k1 + E * k2, cadd(a, t)), x1 = mult(k1 + E * (k2 + PH), csub(a, t));
            if constexpr (INV) {
                const C ai = cadd(x0, x1), bi = cmul(csub(x0, x1), cconj(w));
                const C back = gg ? ai : bi;   // thread 0 keeps the even half (ai), thread 1 the odd (bi)
                C got;
                got.x = __shfl_xor_sync(0xffffffffu, back.x, TW);
                got.y = __shfl_xor_sync(0xffffffffu, back.y, TW);
                u[i] = gg ? got : ai;
                u[HH + i] = gg ? bi : got;
            }
        }
        if constexpr (INV) {
            SmallDFT<PH, +1, C>::run(u);
#pragma unroll
            for (int m = 0; m < PH; ++m) {
                const int l = gg + 2 * m;
                T[cp<real, NY>(c, l, k1)] = cmul(u[m], cconj(tab<G::TABS>(tb.twt + l * E + k1)));
            }
        }
    }
    if constexpr (INV) {
        __syncthreads();
#pragma unroll
        for (int k1 = 0; k1 < E; ++k1) v[k1] = T[cp<real, NY>(c, jl, k1)];
        SmallDFT<E, +1, C>::run(v);
    }
    return true;
}

template <typename real, int NY>
__global__ void __launch_bounds__(Col<real, NY>::NT, col_minb<real, NY>()) kcol_reg(const __grid_constant__ ColArgs<real> A) {
    using G = Col<real, NY>;
    using C = typename G::C;
    constexpr int E = G::E, P = G::P, TW = G::TW;
    extern __shared__ __align__(128) unsigned char col_smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    C *T = reinterpret_cast<C *>(col_smem_raw);   // [NY][TW]
    const ColTab<real, NY> tb(T, A.tab);
    const int h = A.h, tid = threadIdx.x, c = tid % TW, jl = tid / TW;
    const int ntiles = h / TW;
    const int job = (int)blockIdx.x, g = job / ntiles, t = job - g * ntiles;   // (grid.y: run)
    const size_t slot = (size_t)NY * h;
    const ColGroup<real> &gr = A.g[g];
    C *spec = A.spec + (size_t)blockIdx.y * NSLOT * slot + t * TW + c;
    // (no slot is both read and written by different columns of one launch)
    const C *__restrict__ in =
        gr.from_f ? A.f + ((size_t)blockIdx.y * Q + gr.in) * slot + t * TW + c : spec + (size_t)gr.in * slot;
    ColTab<real, NY>::issue(T, A.tab, &bar);
    grid_dep_wait();   // (see kernels_row.cuh)
    C v[E];
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = in[(size_t)(jl + P * q) * h];
    const real mx = gr.c0 * __ldg(A.kx + t * TW + c), c1 = gr.c1, c3 = gr.c3;
    const bool ok = col_pass<real, NY, true>(v, T, tb, &bar, A.err, c, jl, [&](int k, C u) {
        const real ay = tab<G::TABS>(tb.ky + k);
        if (c3 != real(0)) return cscale(u, c3 * ay * ay);   // uniform over the block
        const real m = mx + c1 * ay;
        return C{-m * u.y, m * u.x};
    });
    if (!ok) return;
    C *out = spec + (size_t)gr.out * slot;
#pragma unroll
    for (int q = 0; q < E; ++q) out[(size_t)(jl + P * q) * h] = v[q];
}

// D_y of caller fields g[field][ny][nx] (fp64) into out[2 field + 1] (see
// dx_row; grid: (tiles, fields)), the columns taken two real ones at a time as
// in the stage.
template <typename real, int NY>
__global__ void __launch_bounds__(Col<real, NY>::NT, col_minb<real, NY>()) dy_col(const __grid_constant__ GradArgs<real> A) {
    using G = Col<real, NY>;
    using C = typename G::C;
    constexpr int E = G::E, P = G::P, TW = G::TW;
    extern __shared__ __align__(128) unsigned char col_smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    C *T = reinterpret_cast<C *>(col_smem_raw);
    const ColTab<real, NY> tb(T, A.ctab);
    const int h = A.h, c = threadIdx.x % TW, jl = threadIdx.x / TW;
    const size_t slot = (size_t)NY * h, at = (size_t)blockIdx.x * TW + c;
    const double2 *__restrict__ in = A.g + (size_t)blockIdx.y * slot + at;
    ColTab<real, NY>::issue(T, A.ctab, &bar);
    C v[E];
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const double2 x = in[(size_t)(jl + P * q) * h];
        v[q] = C{(real)x.x, (real)x.y};
    }
    const real s = real(1.0 / NY);
    const bool ok = col_pass<real, NY, true>(v, T, tb, &bar, A.err, c, jl, [&](int k, C u) {
        const real m = tab<G::TABS>(tb.ky + k) * s;
        return C{-m * u.y, m * u.x};
    });
    if (!ok) return;
    double2 *out = A.out + (2 * (size_t)blockIdx.y + 1) * slot + at;
#pragma unroll
    for (int q = 0; q < E; ++q) out[(size_t)(jl + P * q) * h] = make_double2((double)v[q].x, (double)v[q].y);
}
template <typename real, int NY>
__global__ void __launch_bounds__(128) dy_line(const __grid_constant__ GradArgs<real> A) {
    using C = typename cplx_of<real>::type;
    const int h = A.h, kx = (int)blockIdx.x * 128 + (int)threadIdx.x;
    if (kx >= h) return;
    const size_t slot = (size_t)NY * h;
    const double2 *in = A.g + (size_t)blockIdx.y * slot + kx;
    C v[NY];
#pragma unroll
    for (int y = 0; y < NY; ++y) {
        const double2 x = in[(size_t)y * h];
        v[y] = C{(real)x.x, (real)x.y};
    }
    SmallDFT<NY, -1, C>::run(v);
#pragma unroll
    for (int k = 0; k < NY; ++k) {
        const real m = __ldg(A.ky + k) * real(1.0 / NY);
        v[k] = C{-m * v[k].y, m * v[k].x};
    }
    SmallDFT<NY, +1, C>::run(v);
    double2 *out = A.out + (2 * (size_t)blockIdx.y + 1) * slot + kx;
#pragma unroll
    for (int y = 0; y < NY; ++y) out[(size_t)y * h] = make_double2((double)v[y].x, (double)v[y].y);
}

// Sum over the tile's columns of (D_y rho)^2 by Parseval's relation, from the
// real field rho two columns at a time: with Z the transform of f + i f',
// sum_y (D_y f)^2 + (D_y f')^2 = (1 / ny) sum_k k_y^2 |Z_k|^2 (no inverse).
// partial[block]: fp64.
template <typename real, int NY>
__global__ void __launch_bounds__(Col<real, NY>::NT, col_minb<real, NY>()) energy_col(const __grid_constant__ EnergyArgs<real> A) {
    using G = Col<real, NY>;
    using C = typename G::C;
    constexpr int E = G::E, P = G::P, TW = G::TW;
    extern __shared__ __align__(128) unsigned char col_smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    C *T = reinterpret_cast<C *>(col_smem_raw);
    const ColTab<real, NY> tb(T, A.ctab);
    const int h = A.h, c = threadIdx.x % TW, jl = threadIdx.x / TW;
    const C *__restrict__ in = A.rho + (size_t)blockIdx.x * TW + c;
    ColTab<real, NY>::issue(T, A.ctab, &bar);
    grid_dep_wait();
    C v[E];
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = in[(size_t)(jl + P * q) * h];
    double e = 0;
    const bool ok = col_pass<real, NY, false>(v, T, tb, &bar, A.err, c, jl, [&](int k, C u) {
        const real m = tab<G::TABS>(tb.ky + k);
        e += (double)(m * m * (u.x * u.x + u.y * u.y));
        return u;
    });
    if (!ok) return;
    block_sum_store<Col<real, NY>::NT>(e * (1.0 / NY), A.partial_y + blockIdx.x);
}
template <typename real, int NY>
__global__ void __launch_bounds__(128) energy_line(const __grid_constant__ EnergyArgs<real> A) {
    using C = typename cplx_of<real>::type;
    const int h = A.h, kx = (int)blockIdx.x * 128 + (int)threadIdx.x;
    double e = 0;
    grid_dep_wait();
    if (kx < h) {
        C v[NY];
#pragma unroll
        for (int y = 0; y < NY; ++y) v[y] = A.rho[(size_t)y * h + kx];
        SmallDFT<NY, -1, C>::run(v);
#pragma unroll
        for (int k = 0; k < NY; ++k) {
            const real m = __ldg(A.ky + k);
            e += (double)(m * m * (v[k].x * v[k].x + v[k].y * v[k].y));
        }
    }
    block_sum_store<128>(e * (1.0 / NY), A.partial_y + blockIdx.x);
}

// One column of a short grid per thread.
template <typename real, int NY>
__global__ void __launch_bounds__(128) kcol_line(const __grid_constant__ ColArgs<real> A) {
    using C = typename cplx_of<real>::type;
    grid_dep_wait();
    const int h = A.h, ncol = A.ngroups * h;
    const int i = (int)blockIdx.x * 128 + (int)threadIdx.x;
    if (i >= ncol) return;
    const int g = i / h, kx = i - g * h;
    const size_t slot = (size_t)NY * h;
    const ColGroup<real> &gr = A.g[g];
    C *spec = A.spec + (size_t)blockIdx.y * NSLOT * slot + kx;
    const C *in = gr.from_f ? A.f + ((size_t)blockIdx.y * Q + gr.in) * slot + kx : spec + (size_t)gr.in * slot;
    C v[NY];
#pragma unroll
    for (int y = 0; y < NY; ++y) v[y] = in[(size_t)y * h];
    SmallDFT<NY, -1, C>::run(v);
    const real mx = gr.c0 * __ldg(A.kx + kx);
#pragma unroll
    for (int k = 0; k < NY; ++k) {
        const real ay = __ldg(A.ky + k);
        if (gr.c3 != real(0)) {
            v[k] = cscale(v[k], gr.c3 * ay * ay);
        } else {
            const real m = mx + gr.c1 * ay;
            v[k] = C{-m * v[k].y, m * v[k].x};
        }
    }
    SmallDFT<NY, +1, C>::run(v);
    C *out = spec + (size_t)gr.out * slot;
#pragma unroll
    for (int y = 0; y < NY; ++y) out[(size_t)y * h] = v[y];
}

template <typename real, int NY> ColSet col_set() {
    ColSet s;
    if constexpr (NY <= 12) {
        s.k = (const void *)&kcol_line<real, NY>;
        s.dy = (const void *)&dy_line<real, NY>;
        s.energy = (const void *)&energy_line<real, NY>;
        s.nt = 128;
        s.tw = 0;
    } else {
        s.k = (const void *)&kcol_reg<real, NY>;
        s.dy = (const void *)&dy_col<real, NY>;
        s.energy = (const void *)&energy_col<real, NY>;
        s.nt = Col<real, NY>::NT;
        s.tw = Col<real, NY>::TW;
        s.smem = (size_t)NY * s.tw * 2 * sizeof(real) + (Col<real, NY>::TABS ? col_table_bytes<real>(NY, Col<real, NY>::P) : 0);
    }
    return s;
}

}  // namespace ck

}  // namespace fftlb

// Warp-resident row transforms and the fp32 row kernels built on them
// (arXiv:1011.3582, Sec. 3.6, Fig. 3: transform, multiply, inverse).
//
// A row of H = E * P complex values (a real row of 2H values packed as
// z[m] = x[2m] + i x[2m+1]) is transformed by a group of P lanes of one
// warp, in place in shared memory, with no block barrier:
//   stage 1: lane l holds x[l + P t] (t < E) in registers and takes the
//            E-point DFT over t, then multiplies output k1 by W_H^(l k1);
//   transpose: every lane stores its E values at swizzled positions of the
//            same row buffer (__syncwarp before and after);
//   stage 2: the P-point DFTs over l, one per k1, in registers: for P <= E
//            lane j holds the P values of k1 = j + P q (q < E / P); for
//            P = 2E (H = 512) lane k1 + E g holds the even (g = 0) or odd
//            (g = 1) half of the l values, takes an E-point DFT and the
//            last radix-2 step is one exchange with lane ^ E (__shfl_xor);
//   result:  X[k1 + E k2] back in natural order.
// With n = l + P t and k = k1 + E k2, W_H^(nk) = W_H^(l k1) W_P^(l k2)
// W_E^(t k1), which is the decomposition above.  Every index is a
// compile-time constant plus the lane's own offset, and the swizzles keep
// the shared-memory accesses free of bank conflicts for the P >= 16
// layouts (the row groups of P = 8 share banks two ways).
#pragma once

#include "fft_small.cuh"
#include "kernels_pipe.cuh"
#include "row_kernels.h"

namespace fftlb {

// Row configurations: H = E * P, P lanes per row, 32 / P rows per warp
template <int H> struct RowCfg;
template <> struct RowCfg<512> { static constexpr int E = 16, P = 32; };
template <> struct RowCfg<256> { static constexpr int E = 16, P = 16; };
template <> struct RowCfg<128> { static constexpr int E = 16, P = 8; };
// (the cluster rows' lanes: both families read one table of stage-1 twiddles)
static_assert(RowCfg<512>::P == row_p(4, 512) && RowCfg<256>::P == row_p(4, 256) && RowCfg<128>::P == row_p(4, 128), "lanes a row");

// Threads per block: 4 sites of a row each, i.e. 8 row groups and chunks of one
// ring of velocities at every length, and as many blocks on an SM as 128
// registers a thread allow.  Few large blocks with more rows in a chunk wait for
// their own copies and barriers: 512 threads a block at nx = 512 and 256 at nx =
// 256 took K1, K3, K5 27, 23, 47 us on 512^2 (here 23, 16, 32) and 45, 35, 77 on
// 256x2048 (45, 29, 59); 512 threads at nx = 1024 83, 46, 146 on 1024^2 (61, 40,
// 104).
template <int H> __host__ __device__ constexpr int nt_wr() { return H / 2; }
inline int nt_wr_host(int H) { return H / 2; }

// position of stage-1 output (l, k1) in the row buffer.  P >= 16: k1 P +
// (l ^ (k1 mod P)) (for P = 2E, k1 < E: k1 P + (l ^ k1)); P = 8: the row
// parity rsw also flips bit 0 of k1, so that the two rows of a half-warp use
// different banks
template <int H>
__device__ __forceinline__ int tpos(int l, int k1, int rsw) {
    constexpr int P = RowCfg<H>::P;
    return ((k1 ^ rsw) * P) + (l ^ (k1 & (P - 1)));
}

// the lanes of this lane's row group (P consecutive lanes)
template <int P>
__device__ __forceinline__ unsigned group_mask() {
    if constexpr (P >= 32) return 0xffffffffu;
    else return ((1u << P) - 1u) << ((threadIdx.x & 31) & ~(P - 1));
}

// In-place DFT (DIR = -1) or unnormalised inverse (DIR = +1) of the H
// complex values at z by lane j (0 <= j < P) of its row group; tw[k1 P + l]
// = exp(-2 pi i l k1 / H); rsw: row parity (P = 8), else 0.  All P lanes of
// the row group must call it together (they synchronise with __syncwarp on
// the group's mask; other row groups of the warp may diverge).
template <int H, int DIR, typename C>
__device__ __forceinline__ void row_fft_wr(C *z, const C *tw, int j, int rsw) {
    constexpr int E = RowCfg<H>::E, P = RowCfg<H>::P;
    const unsigned gm = group_mask<P>();
    C v[E];
#pragma unroll
    for (int t = 0; t < E; ++t) v[t] = z[j + P * t];
    SmallDFT<E, DIR, C>::run(v);
#pragma unroll
    for (int k1 = 1; k1 < E; ++k1) {
        C w = tw[k1 * P + j];
        if (DIR > 0) w.y = -w.y;
        v[k1] = cmul(v[k1], w);
    }
    __syncwarp(gm);
#pragma unroll
    for (int k1 = 0; k1 < E; ++k1) z[tpos<H>(j, k1, rsw)] = v[k1];
    __syncwarp(gm);
    if constexpr (P <= E) {
        constexpr int NQ = E / P;
        C u[NQ][P];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
#pragma unroll
            for (int l = 0; l < P; ++l) u[q][l] = z[tpos<H>(l, j + P * q, rsw)];
            SmallDFT<P, DIR, C>::run(u[q]);
        }
        __syncwarp(gm);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int k2 = 0; k2 < P; ++k2) z[j + P * q + E * k2] = u[q][k2];
    } else {
        static_assert(P == 2 * E, "row configuration");
        using R = decltype(v[0].x);
        constexpr int HE = E / 2;
        const int k1 = j & (E - 1), g = j / E;
        C u[E];
#pragma unroll
        for (int m = 0; m < E; ++m) u[m] = z[tpos<H>(g + 2 * m, k1, 0)];
        SmallDFT<E, DIR, C>::run(u);
        // X[k1 + E (k2' + E k3)] = V0[k2'] + (-1)^k3 W_P^k2' V1[k2']: lane
        // g keeps k2' in [HE g, HE g + HE) and receives the other lane's half
        C a[HE], b[HE];
#pragma unroll
        for (int i = 0; i < HE; ++i) {
            const C send = g ? u[i] : u[HE + i];
            C recv;
            recv.x = __shfl_xor_sync(0xffffffffu, send.x, E);
            recv.y = __shfl_xor_sync(0xffffffffu, send.y, E);
            a[i] = g ? recv : u[i];
            b[i] = g ? u[HE + i] : recv;
        }
        __syncwarp(gm);   // every lane's stage-2 reads are done
#pragma unroll
        for (int i = 0; i < HE; ++i) {
            R c, s;
            w32<DIR, R>(i, c, s);   // W_P^i, P = 32
            C t = i == 0 ? b[i] : C{b[i].x * c - b[i].y * s, b[i].x * s + b[i].y * c};
            // times W_P^(HE g): W_32^8 = -i forward, +i inverse
            const C r = DIR < 0 ? cmul_mi(t) : cmul_i(t);
            t = g ? r : t;
            const int k2 = HE * g + i;
            z[k1 + E * k2] = cadd(a[i], t);
            z[k1 + E * (k2 + E)] = csub(a[i], t);
        }
        __syncwarp(gm);
        return;
    }
    __syncwarp(gm);
}

// Forward real rows: the natural-order result Z of row_fft_wr (the
// half-length transform of the packed row) -> one-sided spectrum X[0 .. H-1]
// with the real Nyquist value in the imaginary part of X[0], written to
// out (global memory, coalesced: lanes take consecutive k and H - k).
// Wh[k] = exp(-2 pi i k / 2H) / 2, k < H / 2.
template <int H, typename C>
__device__ __forceinline__ void r2c_post_wr(const C *z, C *out, const C *Wh, int j) {
    using R = decltype(z[0].x);
    constexpr int P = RowCfg<H>::P;
#pragma unroll
    for (int k0 = 0; k0 < H / 2; k0 += P) {
        const int k = k0 + j;
        if (k == 0) {
            const C z0 = z[0];
            out[0] = C{z0.x + z0.y, z0.x - z0.y};
            out[H / 2] = cconj(z[H / 2]);
        } else {
            const C p = z[k], q = z[H - k];
            const C s = cadd(p, cconj(q)), w = cmul(Wh[k], cmul_mi(csub(p, cconj(q))));
            out[k] = C{R(0.5) * s.x + w.x, R(0.5) * s.y + w.y};
            out[H - k] = C{R(0.5) * s.x - w.x, w.y - R(0.5) * s.y};
        }
    }
}

// r2c_post_wr times i k_x c: dst[k] = i kxt[k] sx X[k] (bin 0, DC and
// row-Nyquist, has k_x = 0 for both).  dst may be z.
template <int H, typename C>
__device__ __forceinline__ void r2c_post_dx(const C *z, C *dst, const float *__restrict__ kxt, float sx, const C *Wh,
                                            int j) {
    using R = decltype(z[0].x);
    constexpr int P = RowCfg<H>::P;
#pragma unroll
    for (int k0 = 0; k0 < H / 2; k0 += P) {
        const int k = k0 + j;
        if (k == 0) {
            dst[0] = C{0, 0};
            dst[H / 2] = imul(kxt[H / 2] * sx, cconj(z[H / 2]));
        } else {
            const C p = z[k], q = z[H - k];
            const C s = cadd(p, cconj(q)), w = cmul(Wh[k], cmul_mi(csub(p, cconj(q))));
            dst[k] = imul(kxt[k] * sx, C{R(0.5) * s.x + w.x, R(0.5) * s.y + w.y});
            dst[H - k] = imul(kxt[H - k] * sx, C{R(0.5) * s.x - w.x, w.y - R(0.5) * s.y});
        }
    }
}

// Inverse real rows, in place: one-sided packed spectrum X -> Z[k] = (X[k]
// + X[k + H]) + i (X[k] - X[k + H]) exp(+2 pi i k / 2H), X[k + H] =
// conj X[H - k]; the half-length inverse of Z is the real row.
template <int H, typename C>
__device__ __forceinline__ void c2r_pre_wr(C *z, const C *Wp, int j) {
    using R = decltype(z[0].x);
    constexpr int P = RowCfg<H>::P;
#pragma unroll
    for (int k0 = 0; k0 < H / 2; k0 += P) {
        const int k = k0 + j;
        if (k == 0) {
            const C x0 = z[0];
            z[0] = C{x0.x + x0.y, x0.x - x0.y};
            const C xh = z[H / 2];   // Z = 2 conj X
            z[H / 2] = C{R(2) * xh.x, R(-2) * xh.y};
        } else {
            // with a = p + conj q, e = i (p - conj q) conj w: Z[k] = a + e,
            // Z[H - k] = conj(a - e)
            const C p = z[k], q = z[H - k];
            const C a = cadd(p, cconj(q)), e = cmul_i(cmul(csub(p, cconj(q)), cconj(Wp[k])));
            z[k] = cadd(a, e);
            z[H - k] = cconj(csub(a, e));
        }
    }
}

// four consecutive floats (16-byte aligned) to and from registers
__device__ __forceinline__ void ld4(float (&a)[4], const float *p) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    a[0] = v.x;
    a[1] = v.y;
    a[2] = v.z;
    a[3] = v.w;
}
__device__ __forceinline__ void st4(float *p, const float (&a)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(a[0], a[1], a[2], a[3]);
}
// ... of values that leave the L2 first: f^n and the new f are not read again
// before the spectra are (1024^2: K5 107.6 -> 106.2 us)
__device__ __forceinline__ void ld4_once(float (&a)[4], const float *p) {
    const float4 v = __ldcs(reinterpret_cast<const float4 *>(p));
    a[0] = v.x;
    a[1] = v.y;
    a[2] = v.z;
    a[3] = v.w;
}
__device__ __forceinline__ void st4_once(float *p, const float (&a)[4]) {
    __stcs(reinterpret_cast<float4 *>(p), make_float4(a[0], a[1], a[2], a[3]));
}

// ---------------------------------------------------------------------------
// K1 (fp32, nx = 2H): moments rho, u, T (Eqs. 7-9), the level-1 fields
// Pi = P^w - rho T (Eq. 18) and g = M/T, and the forward row transforms of
// the 24 f_i with v_x != 0 and of rho, u_x, u_y, T, Pi, g, as k1_pipe, with
// warp-resident row transforms.  Persistent over the rows of all runs;
// per row, 32 / NG chunks of distribution rows (the first also holds the
// rest velocity's row, which only enters the moments), NG = rows per block
// pass (one per row group), two chunk buffers.
// ---------------------------------------------------------------------------

// the distribution rows of chunk c of a row: the rest velocity and the
// first NG moving rows, then NG moving rows per chunk
__host__ __device__ constexpr int k1w_first(int c, int NG) { return c == 0 ? 0 : 1 + c * NG; }
__host__ __device__ constexpr int k1w_count(int c, int NG) { return c == 0 ? NG + 1 : NG; }

__device__ __forceinline__ void k1w_issue(const float *f, float *dst, uint64_t *bar, int j, int nchunk, int NG,
                                          int nx, int ny, size_t N) {
    const int ri = j / nchunk, c = j - ri * nchunk;
    const int yg = (int)blockIdx.x + ri * (int)gridDim.x;   // row over all runs
    const int run = yg / ny, y = yg - run * ny;
    const int i0 = k1w_first(c, NG), nf = k1w_count(c, NG);
    const uint32_t rowbytes = (uint32_t)(nx * sizeof(float));
    const float *fr = f + (size_t)run * Q * N;
    mbar_expect_tx(bar, (uint32_t)nf * rowbytes);
    for (int r = 0; r < nf; ++r)
        bulk_g2s(dst + (size_t)r * nx, fr + (size_t)(i0 + r) * N + (size_t)y * nx, rowbytes, bar);
}

template <int H>
__global__ void __launch_bounds__(nt_wr<H>(), 512 / nt_wr<H>()) k1_wr(const float *f, float2 *spec, float *__restrict__ fields,
                                                 const float2 *__restrict__ tw_g, const float2 *__restrict__ Wh_g,
                                                 const float *__restrict__ kxt, KP<float> P, int *err) {
    using C = float2;
    using real = float;
    constexpr int NX = 2 * H, NT = nt_wr<H>(), NWARP = NT / 32;
    constexpr int PL = RowCfg<H>::P, RPW = 32 / PL;
    constexpr int NG = NWARP * RPW;                // row groups per block
    constexpr int CH = NG + 1, NCH = NMOV / NG;    // rows per chunk buffer, chunks per row
    constexpr int SMAX = NX / NT;
    static_assert(NMOV % NG == 0 && NG % 8 == 0, "chunking");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar0, bar1;
    const int nx = NX, ny = P.ny, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = warp * RPW + lane / PL, j = lane & (PL - 1);
    const int rsw = PL == 8 ? ((lane / PL) & 1) : 0;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    SmemCursor sc{smem_raw, 0u};
    C *tw = (C *)sc.take(H * sizeof(C));
    C *Wh = (C *)sc.take(H / 2 * sizeof(C));
    real *kxs = (real *)sc.take(H * sizeof(real));   // k_x of the row bins
    real *buf0 = (real *)sc.take((size_t)CH * NX * sizeof(real));
    real *buf1 = (real *)sc.take((size_t)CH * NX * sizeof(real));
    real *fb = (real *)sc.take((size_t)6 * NX * sizeof(real));   // rho, ux, uy, T, Pi, g rows
    const int NY = P.nrun * ny;
    const int nrows = (int)blockIdx.x < NY ? (NY - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int njobs = nrows * NCH;
    if (tid == 0) {   // (the first copies start while the tables load)
        mbar_init(&bar0, 1);
        mbar_init(&bar1, 1);
        mbar_init_fence();
        grid_dep_wait();
        if (njobs > 0) k1w_issue(f, buf0, &bar0, 0, NCH, NG, nx, ny, N);
        if (njobs > 1) k1w_issue(f, buf1, &bar1, 1, NCH, NG, nx, ny, N);
    }
    load_tab4(tw, tw_g, H, NT);
    load_tab4(Wh, Wh_g, H / 2, NT);
    load_tab4(kxs, kxt, H, NT);
    grid_dep_wait();
    __syncthreads();
    uint32_t par0 = 0, par1 = 0;
    bool pend0 = njobs > 0, pend1 = njobs > 1;
    real a0[SMAX], a1[SMAX], a2[SMAX], a3[SMAX];
#pragma unroll
    for (int s = 0; s < SMAX; ++s) a0[s] = a1[s] = a2[s] = a3[s] = real(0);
    for (int jb = 0; jb < njobs; ++jb) {
        const bool odd = jb & 1;
        uint64_t *bar = odd ? &bar1 : &bar0;
        const int ri = jb / NCH, c = jb - ri * NCH;
        const int yg = (int)blockIdx.x + ri * (int)gridDim.x;
        const int run = yg / ny, y = yg - run * ny;
        C *spec_r = spec + (size_t)run * NSLOT * slot;
        real *fields_r = fields + (size_t)run * NSLOT * N;
        const int i0 = k1w_first(c, NG), nf = k1w_count(c, NG);
        if (!block_wait(bar, odd ? par1 : par0, err)) {
            if (pend0) mbar_wait_bounded(&bar0, par0);
            if (pend1) mbar_wait_bounded(&bar1, par1);
            return;
        }
        if (odd) {
            par1 ^= 1;
            pend1 = false;
        } else {
            par0 ^= 1;
            pend0 = false;
        }
        real *B = odd ? buf1 : buf0;
        // moments (Eqs. 7-9): sums over this chunk's rows, ring by ring (speed
        // s_k, directions r pi / 4), 19 operations a ring and site
        const int q0 = c == 0 ? 1 : 0;   // chunk row of the first ring's direction 0
#pragma unroll
        for (int s = 0; s < SMAX; ++s) {
            const int x = tid + s * NT;
            if (c == 0) a0[s] += B[x];   // the rest velocity
#pragma unroll 1
            for (int rr = 0; rr < NG / 8; ++rr) {
                const real *q = B + (size_t)(q0 + 8 * rr) * NX + x;
                const int v0 = 1 + c * NG + 8 * rr;
                real v[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) v[r] = q[(size_t)r * NX];
                const real sum = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
                const real d15 = v[1] - v[5], d37 = v[3] - v[7], hh = real(0.70710678118654752440);
                a0[s] += sum;
                a1[s] += VX<real>(v0) * ((v[0] - v[4]) + hh * (d15 - d37));
                a2[s] += VX<real>(v0) * ((v[2] - v[6]) + hh * (d15 + d37));
                a3[s] += V2<real>(v0) * sum;
            }
        }
        __syncthreads();
        // forward transforms of the chunk's moving rows: group grp takes
        // chunk row grp + (c == 0) (the first chunk's row 0 is the rest
        // velocity), i.e. f_i with i = i0 + that row, into slot i - 1
        {
            const int r = grp + (c == 0 ? 1 : 0);
            // (v_x = 0: the column pass takes f_i itself)
            if (r < nf && VX<real>(i0 + r) != real(0)) {
                const int i = i0 + r;
                C *zr = reinterpret_cast<C *>(B) + (size_t)r * H;
                C *dst = spec_r + (size_t)(i - 1) * slot + (size_t)y * H;
                row_fft_wr<H, -1>(zr, tw, j, rsw);
                if (VY<real>(i) == real(0))   // convection in k_x alone: i v_x k_x f^ / nx, no column pass
                    r2c_post_dx<H>(zr, dst, kxs, VX<real>(i) * P.scale_x, Wh, j);
                else
                    r2c_post_wr<H>(zr, dst, Wh, j);
            }
        }
        if (c == NCH - 1) {
            // the level-1 fields of this row, then their forward transforms
#pragma unroll
            for (int s = 0; s < SMAX; ++s) {
                const int x = tid + s * NT;
                const real rho = a0[s], ux = a1[s] / rho, uy = a2[s] / rho;
                const real T = real(0.5) * (a3[s] / rho - (ux * ux + uy * uy));
                const size_t o = (size_t)y * nx + x;
                fields_r[o] = rho;
                fields_r[N + o] = ux;
                fields_r[2 * N + o] = uy;
                fields_r[3 * N + o] = T;
                fb[x] = rho;
                fb[NX + x] = ux;
                fb[2 * NX + x] = uy;
                fb[3 * NX + x] = T;
                const real Pi = rho * T / (real(1) - P.b * rho) - P.a * rho * rho - rho * T;   // Eq. 18
                const real g = (P.K + P.H * T) / T;                                          // M / T
                fields_r[4 * N + o] = Pi;
                fields_r[5 * N + o] = g;
                fb[4 * NX + x] = Pi;
                fb[5 * NX + x] = g;
                a0[s] = a1[s] = a2[s] = a3[s] = real(0);
            }
            __syncthreads();
            if (grp < 6) {
                C *zr = reinterpret_cast<C *>(fb) + (size_t)grp * H;
                row_fft_wr<H, -1>(zr, tw, j, rsw);
                r2c_post_wr<H>(zr, spec_r + (size_t)(SLOT_RHO + grp) * slot + (size_t)y * H, Wh, j);
            }
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0 && jb + 2 < njobs) {   // job jb + 2 reuses this buffer
            k1w_issue(f, B, bar, jb + 2, NCH, NG, nx, ny, N);
            if (odd) pend1 = true;
            else pend0 = true;
        }
    }
}

// shared memory of k1_wr<H>
inline size_t k1_wr_smem(int H) {
    const int P = H == 512 ? 32 : H == 256 ? 16 : 8;
    const int CH = nt_wr_host(H) / P + 1;
    return smem_bytes({(size_t)H * 8, (size_t)H / 2 * 8, (size_t)H * 4, (size_t)CH * 2 * H * 4,
                       (size_t)CH * 2 * H * 4, (size_t)6 * 2 * H * 4});
}

// ---------------------------------------------------------------------------
// K3 (fp32, nx = 2H): inverse rows of the 11 level-1 derivatives that have a
// factor k_x or start from a row spectrum (stage_layout.cuh) -> Lambda (Eq. 19),
// Phi (Eq. 23), the numerators of C (Eq. 22) and B (Eq. 21) -> d_x of Lambda_xx,
// Lambda_xy, Phi_x (a forward and an inverse row each) added to the numerators.
// Persistent over the rows of all runs, one row per pass and one buffer of the 11
// transformed rows; the 8 real rows are read where they are used, from the L2
// they were sent to with the row's copies, which leaves room and registers for a
// third block on the SM (all 19 rows staged, two blocks: 39.6 us on 1024^2, 73.6
// on 1024x2048; so 36.8 and 65.5).
// ---------------------------------------------------------------------------

// the row's spectra into dst, its real rows into L2
template <typename C>
__device__ __forceinline__ void k3_issue(const C *spec, C *dst, uint64_t *bar, int ri, int ny, size_t slot, int h) {
    const int yg = (int)blockIdx.x + ri * (int)gridDim.x;
    const int run = yg / ny, y = yg - run * ny;
    spec += (size_t)run * NSLOT * slot + (size_t)y * h;
    const uint32_t rowbytes = (uint32_t)(h * sizeof(C));
    mbar_expect_tx(bar, (uint32_t)(NSP - 3) * rowbytes);   // D_LAP, D_DIVX, D_DIVY are formed in K3
    for (int o = 0; o < NSP; ++o)
        if (k3_src_slot(o) >= 0) bulk_g2s(dst + (size_t)o * h, spec + (size_t)k3_src_slot(o) * slot, rowbytes, bar);
    for (int o = NSP; o < NK3; ++o) bulk_prefetch_l2(spec + (size_t)k3_src_slot(o) * slot, rowbytes);
}

template <int H>
__global__ void __launch_bounds__(nt_wr<H>(), 768 / nt_wr<H>()) k3_wr(float2 *spec, const float2 *__restrict__ tw_g,
                                                 const float2 *__restrict__ Wp_g, const float2 *__restrict__ Wh_g,
                                                 const float *__restrict__ kxt,
                                                 KP<float> P, int *err) {
    using C = float2;
    using real = float;
    constexpr int NX = 2 * H, NT = nt_wr<H>();
    constexpr int PL = RowCfg<H>::P, RPW = 32 / PL, NG = (NT / 32) * RPW;   // row groups
    constexpr int SMAX = NX / NT;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    const int ny = P.ny, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = warp * RPW + lane / PL, j = lane & (PL - 1);
    const int rsw = PL == 8 ? ((lane / PL) & 1) : 0;
    const size_t slot = (size_t)ny * H;
    SmemCursor sc{smem_raw, 0u};
    C *tw = (C *)sc.take(H * sizeof(C));
    C *Wp = (C *)sc.take(H / 2 * sizeof(C));
    C *Wh = (C *)sc.take(H / 2 * sizeof(C));
    real *kxs = (real *)sc.take(H * sizeof(real));   // k_x of the row bins
    C *dc = (C *)sc.take((size_t)NSP * H * sizeof(C));
    const int NY = P.nrun * ny;
    const int nrows = (int)blockIdx.x < NY ? (NY - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    if (tid == 0) {   // (the first copies start before the tables load)
        mbar_init(&bar, 1);
        mbar_init_fence();
        grid_dep_wait();
        if (nrows > 0) k3_issue(spec, dc, &bar, 0, ny, slot, H);
    }
    load_tab4(tw, tw_g, H, NT);
    load_tab4(Wp, Wp_g, H / 2, NT);
    load_tab4(Wh, Wh_g, H / 2, NT);
    load_tab4(kxs, kxt, H, NT);
    grid_dep_wait();
    __syncthreads();
    for (int ri = 0; ri < nrows; ++ri) {
        const int yg = (int)blockIdx.x + ri * (int)gridDim.x;
        const int run = yg / ny, y = yg - run * ny;
        C *spec_r = spec + (size_t)run * NSLOT * slot + (size_t)y * H;
        if (!block_wait(&bar, ri & 1, err)) {
            mbar_wait_bounded(&bar, ri & 1);
            return;
        }
        for (int k = tid; k < H; k += NT) k3_form_x<real>(dc, H, k, kxs[k], P.scale_x);
        __syncthreads();
        for (int r = grp; r < NSP; r += NG) {   // (uniform over each row group)
            C *zr = dc + (size_t)r * H;
            c2r_pre_wr<H>(zr, Wp, j);
            __syncwarp(group_mask<PL>());
            row_fft_wr<H, +1>(zr, tw, j, rsw);
        }
        __syncthreads();
        auto out = [&](int s) { return reinterpret_cast<real *>(spec_r + (size_t)s * slot); };
#pragma unroll 1
        for (int s = 0; s < SMAX; s += 2) {   // two consecutive sites
            const int x = 2 * tid + s * NT;
            float2 v[NK3];
#pragma unroll
            for (int o = NSP; o < NK3; ++o)
                v[o] = *reinterpret_cast<const float2 *>(out(k3_src_slot(o)) + x);
#pragma unroll
            for (int o = 0; o < NSP; ++o) v[o] = dc[o * H + (x >> 1)];
            const Level2<real> l = level2_site<real>([&](int o) { return v[o].x; }, P);
            const Level2<real> m = level2_site<real>([&](int o) { return v[o].y; }, P);
            auto st = [&](int q, real a, real b) { *reinterpret_cast<float2 *>(out(q) + x) = make_float2(a, b); };
            st(SLOT_L2, l.Lxy, m.Lxy);
            st(SLOT_L2 + 1, l.Lyy, m.Lyy);
            st(SLOT_L2 + 2, l.Phy, m.Phy);
            // rows 0..2: transformed next; 3..5: the numerators their d_x
            // joins (same sites, same thread)
            auto keep = [&](int r, real a, real b) { dc[r * H + (x >> 1)] = make_float2(a, b); };
            keep(0, l.Phx, m.Phx);
            keep(1, l.Lxx, m.Lxx);
            keep(2, l.Lxy, m.Lxy);
            keep(3, l.Cn, m.Cn);
            keep(4, l.Bx, m.Bx);
            keep(5, l.By, m.By);
        }
        __syncthreads();
        for (int r = grp; r < 3; r += NG) {
            C *zr = dc + (size_t)r * H;
            row_fft_wr<H, -1>(zr, tw, j, rsw);
            r2c_post_dx<H>(zr, zr, kxs, P.scale_x, Wh, j);
            __syncwarp(group_mask<PL>());
            c2r_pre_wr<H>(zr, Wp, j);
            __syncwarp(group_mask<PL>());
            row_fft_wr<H, +1>(zr, tw, j, rsw);
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < SMAX; s += 2) {
            const int x = 2 * tid + s * NT;
#pragma unroll
            for (int r = 0; r < 3; ++r)
                *reinterpret_cast<float2 *>(out(SLOT_A + r) + x) = cadd(dc[(3 + r) * H + (x >> 1)], dc[r * H + (x >> 1)]);
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0 && ri + 1 < nrows) k3_issue(spec, dc, &bar, ri + 1, ny, slot, H);
    }
}

// shared memory of k3_wr<H>
inline size_t k3_wr_smem(int H) {
    return smem_bytes({(size_t)H * 8, (size_t)H / 2 * 8, (size_t)H / 2 * 8, (size_t)H * 4, (size_t)NSP * 2 * H * 4});
}

// ---------------------------------------------------------------------------
// K5 (fp32, nx = 2H): convection rows + level-2 divergences (inverse) ->
// A, B, C, C_q (Eqs. 20-23), f^eq (Eq. 3), I (Eq. 11), BGK and the RK
// combination (Eq. 10), as k5_pipe, with warp-resident row transforms.
// Persistent over the rows of all runs; per row: the head (3 level-2
// spectra, rho, u_x, u_y, T, the 3 aux numerators) and 4 chunks of 8 convection
// rows, one ring each (two buffers), one row per row group.
// ---------------------------------------------------------------------------

template <int H>
__global__ void __launch_bounds__(nt_wr<H>(), 512 / nt_wr<H>()) k5_wr(const float2 *spec, const float *fields,
                                                 const float *aux, const float *fcur, const float *fbase,
                                                 float *fout, float alpha, float beta,
                                                 const float2 *__restrict__ tw_g, const float2 *__restrict__ Wp_g,
                                                 KP<float> P, int *err) {
    using C = float2;
    using real = float;
    constexpr int NX = 2 * H, NT = nt_wr<H>();
    constexpr int PL = RowCfg<H>::P, RPW = 32 / PL;          // lanes per row, rows per warp
    constexpr int CH = 8, NCH = NMOV / CH;                     // rows (one ring) per chunk, chunks per row
    static_assert(NX == 4 * NT && NT == CH * PL, "four sites a thread, one row a group");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar0, bar1, hbar;
    const int nx = NX, ny = P.ny, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grow = warp * RPW + lane / PL, j = lane & (PL - 1);   // row within the chunk, lane within the row
    const int rsw = PL == 8 ? ((lane / PL) & 1) : 0;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    SmemCursor sc{smem_raw, 0u};
    C *tw = (C *)sc.take(H * sizeof(C));
    C *Wp = (C *)sc.take(H / 2 * sizeof(C));
    real *Hd = (real *)sc.take((size_t)NHEAD * NX * sizeof(real));
    real *buf0 = (real *)sc.take((size_t)CH * NX * sizeof(real));
    real *buf1 = (real *)sc.take((size_t)CH * NX * sizeof(real));
    const int NY = P.nrun * ny;
    const int nrows = (int)blockIdx.x < NY ? (NY - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int njobs = nrows * NCH;
    if (tid == 0) {   // (the first copies start before the tables load)
        mbar_init(&bar0, 1);
        mbar_init(&bar1, 1);
        mbar_init(&hbar, 1);
        mbar_init_fence();
        grid_dep_wait();
        if (njobs > 0) k5_issue_chunk<real>(spec, buf0, &bar0, 0, NCH, CH, nx, ny, slot, H);
        if (njobs > 1) k5_issue_chunk<real>(spec, buf1, &bar1, 1, NCH, CH, nx, ny, slot, H);
        if (nrows > 0) k5_issue_head<real>(spec, fields, aux, Hd, &hbar, 0, nx, ny, N, slot, H);
    }
    load_tab4(tw, tw_g, H, NT);
    load_tab4(Wp, Wp_g, H / 2, NT);
    __syncthreads();
    uint32_t par0 = 0, par1 = 0;
    bool pend0 = njobs > 0, pend1 = njobs > 1, hpend = nrows > 0;
    const real dt = P.dt, itau = real(1) / P.tau;
    const bool with_base = alpha != real(0);
    for (int jb = 0; jb < njobs; ++jb) {
        const bool odd = jb & 1;
        const int ri = jb / NCH, c = jb - ri * NCH;
        const int yg = (int)blockIdx.x + ri * (int)gridDim.x;
        const int run = yg / ny, y = yg - run * ny;
        const size_t fo = (size_t)run * Q * N;
        if (!block_wait(odd ? &bar1 : &bar0, odd ? par1 : par0, err)) {
            if (pend0) mbar_wait_bounded(&bar0, par0);
            if (pend1) mbar_wait_bounded(&bar1, par1);
            if (hpend) mbar_wait_bounded(&hbar, ri & 1);
            return;
        }
        if (odd) {
            par1 ^= 1;
            pend1 = false;
        } else {
            par0 ^= 1;
            pend0 = false;
        }
        real *B = odd ? buf1 : buf0;
        // inverse transform of convection row grow of the chunk; with the
        // first chunk, then the wait for the head
        {
            // (directions 2 and 6 of a ring, v_x = 0: real from the column pass)
            if ((grow & 3) != 2) {
                C *zr = reinterpret_cast<C *>(B) + (size_t)grow * H;
                c2r_pre_wr<H>(zr, Wp, j);
                __syncwarp(group_mask<PL>());
                row_fft_wr<H, +1>(zr, tw, j, rsw);
            }
            if (c == 0) {
                if (!block_wait(&hbar, ri & 1, err)) {
                    if (pend0) mbar_wait_bounded(&bar0, par0);
                    if (pend1) mbar_wait_bounded(&bar1, par1);
                    mbar_wait_bounded(&hbar, ri & 1);
                    return;
                }
                hpend = false;
            }
        }
        __syncthreads();
        if (c == 0) {
            // per-site coefficients over the head rows (same site, same
            // thread): row 0 <- e0, 1 <- e1x, 2 <- e1y, 7 <- C + C_q, 8 <- 1/T;
            // the rest velocity's update
            const int x0 = 4 * tid;
            const size_t o = fo + (size_t)y * nx + x0;
            real rho[4], ux[4], uy[4], T[4], dLx[4], dLy[4], dPh[4], a7[4], a8[4], a9[4], fc[4], fb[4];
            ld4(rho, Hd + 3 * nx + x0);
            ld4(ux, Hd + 4 * nx + x0);
            ld4(uy, Hd + 5 * nx + x0);
            ld4(T, Hd + 6 * nx + x0);
            ld4(dLx, Hd + x0);
            ld4(dLy, Hd + nx + x0);
            ld4(dPh, Hd + 2 * nx + x0);
            ld4(a7, Hd + 7 * nx + x0);
            ld4(a8, Hd + 8 * nx + x0);
            ld4(a9, Hd + 9 * nx + x0);
            ld4(fc, fcur + o);
            if (with_base) ld4(fb, fbase + o);
            real e0[4], e1x[4], e1y[4], CC[4], iT[4], fn[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const real rT = rho[q] * T[q];
                const real inv2 = real(1) / (real(2) * rho[q] * T[q] * T[q]);
                const real Bx = (a8[q] + dLx[q]) / rT;      // Eq. 21
                const real By = (a9[q] + dLy[q]) / rT;
                CC[q] = (a7[q] + dPh[q]) * inv2;            // C + C_q, Eqs. 22-23
                const real A = real(-2) * CC[q] * T[q];      // Eq. 20
                const real u2 = ux[q] * ux[q] + uy[q] * uy[q];
                e0[q] = A - (Bx * ux[q] + By * uy[q]) + CC[q] * u2;
                e1x[q] = Bx - real(2) * CC[q] * ux[q];
                e1y[q] = By - real(2) * CC[q] * uy[q];
                iT[q] = real(1) / T[q];
                real F[5];
                weights_Fk<real>(T[q], F);
                const real qq = real(0.5) * u2 / T[q], om = real(1) - qq;
                const real fe = rho[q] * F[0] * (om + real(0.5) * qq * qq);
                fn[q] = rk_combine(with_base, beta, dt, fc[q], fb[q], -(fc[q] - fe) * itau - e0[q] * fe);
            }
            st4(Hd + x0, e0);
            st4(Hd + nx + x0, e1x);
            st4(Hd + 2 * nx + x0, e1y);
            st4(Hd + 7 * nx + x0, CC);
            st4(Hd + 8 * nx + x0, iT);
            st4(fout + o, fn);
            __syncthreads();
        }
        // epilogue: ring c (velocities 1 + 8c .. 8 + 8c of Eq. 1, one speed, one
        // weight, the eight directions known at compile time), four consecutive
        // sites per thread: 16-byte loads and stores (1024^2: 126.7 us against
        // 130.9 site by site)
        {
            const int v0 = 8 * c;
            const real sk = VX<real>(1 + v0), sk2 = V2<real>(1 + v0);
            const real *cres = B;
            const int x0 = 4 * tid;
            const size_t o0 = fo + (size_t)(1 + v0) * N + (size_t)y * nx + x0;
            real rho[4], ux[4], uy[4], T[4], iT[4], e0[4], e1x[4], e1y[4], CC[4];
            ld4(rho, Hd + 3 * nx + x0);
            ld4(ux, Hd + 4 * nx + x0);
            ld4(uy, Hd + 5 * nx + x0);
            ld4(T, Hd + 6 * nx + x0);
            ld4(iT, Hd + 8 * nx + x0);
            ld4(e0, Hd + x0);
            ld4(e1x, Hd + nx + x0);
            ld4(e1y, Hd + 2 * nx + x0);
            ld4(CC, Hd + 7 * nx + x0);
            real p0[4], p1[4], p2[4], p3[4], p4[4], h0[4], uxk[4], uyk[4], exk[4], eyk[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const real qq = real(0.5) * (ux[q] * ux[q] + uy[q] * uy[q]) * iT[q], om = real(1) - qq;
                const real rF = rho[q] * weight_Fk<real>(c, T[q]);   // Eq. 4
                const real r1 = rF * iT[q], r2 = r1 * iT[q], r3 = r2 * iT[q];
                p0[q] = rF * (om + real(0.5) * qq * qq);   // rho F_k times the factors of Eq. 3
                p1[q] = r1 * om;
                p2[q] = real(0.5) * r2 * om;
                p3[q] = r3 * (real(1) / real(6));
                p4[q] = r3 * iT[q] * (real(1) / real(24));
                h0[q] = e0[q] + CC[q] * sk2;
                uxk[q] = sk * ux[q];
                uyk[q] = sk * uy[q];
                exk[q] = sk * e1x[q];
                eyk[q] = sk * e1y[q];
            }
            // directions r and r + 4 together: f^eq = even +- odd in v.u;
            // rhs = -(f - f^eq) / tau - g f^eq - convection with g = -I / f^eq
            // (Eqs. 10, 11).  The distributions of two such pairs are
            // loaded before any of their stores, as fout may alias fcur or
            // fbase.
            const real *__restrict__ pc = fcur + o0;
            const real *__restrict__ pb = fbase + o0;
            real *__restrict__ po = fout + o0;
#pragma unroll
            for (int r0 = 0; r0 < 4; r0 += 2) {
                real fc[4][4], fb[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int d = r0 + (r >> 1) + 4 * (r & 1);
                    ld4(fc[r], pc + (size_t)d * N);
                    if (with_base) ld4_once(fb[r], pb + (size_t)d * N);
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    real cv[2][4], fn[2][4];
                    ld4(cv[0], cres + (size_t)(r0 + r) * NX + x0);
                    ld4(cv[1], cres + (size_t)(r0 + r + 4) * NX + x0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const real vu = dir_dot<real>(r0 + r, uxk[q], uyk[q]), w2 = vu * vu;
                        const real ev = p0[q] + w2 * (p2[q] + w2 * p4[q]), od = vu * (p1[q] + w2 * p3[q]);   // Eq. 3
                        const real ed = dir_dot<real>(r0 + r, exk[q], eyk[q]);
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            const real fe = s ? ev - od : ev + od, g = s ? h0[q] - ed : h0[q] + ed;
                            const real f = fc[2 * r + s][q];
                            const real rhs = -(f - fe) * itau - cv[s][q] - g * fe;
                            fn[s][q] = rk_combine(with_base, beta, dt, f, fb[2 * r + s][q], rhs);
                        }
                    }
                    st4_once(po + (size_t)(r0 + r) * N, fn[0]);
                    st4_once(po + (size_t)(r0 + r + 4) * N, fn[1]);
                }
            }
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0 && jb + 1 < njobs) {
            // the next job's distribution rows (current and, for RK stages 2
            // and 3, base state) into L2 ahead of its epilogue's loads
            const int nri = (jb + 1) / NCH, nc = (jb + 1) - nri * NCH;
            const int nyg = (int)blockIdx.x + nri * (int)gridDim.x;
            const int nrun = nyg / ny, ny_ = nyg - nrun * ny;
            const size_t no = (size_t)nrun * Q * N + (size_t)(1 + nc * CH) * N + (size_t)ny_ * nx;
            for (int r = 0; r < CH; ++r) {
                bulk_prefetch_l2(fcur + no + (size_t)r * N, (uint32_t)(NX * sizeof(real)));
                if (with_base) bulk_prefetch_l2(fbase + no + (size_t)r * N, (uint32_t)(NX * sizeof(real)));
            }
        }
        if (tid == 0) {
            if (jb + 2 < njobs) {
                const bool nodd = jb & 1;   // chunk jb + 2 reuses this buffer
                k5_issue_chunk<real>(spec, B, nodd ? &bar1 : &bar0, jb + 2, NCH, CH, nx, ny, slot, H);
                if (nodd) pend1 = true;
                else pend0 = true;
            }
            if (c == NCH - 1 && ri + 1 < nrows) {   // the row's head buffer is free
                k5_issue_head<real>(spec, fields, aux, Hd, &hbar, ri + 1, nx, ny, N, slot, H);
                hpend = true;
            }
        }
    }
}

// shared memory of k5_wr<H>
inline size_t k5_wr_smem(int H) {
    return smem_bytes({(size_t)H * 8, (size_t)H / 2 * 8, (size_t)NHEAD * 2 * H * 4, (size_t)8 * 2 * H * 4, (size_t)8 * 2 * H * 4});
}

}  // namespace fftlb

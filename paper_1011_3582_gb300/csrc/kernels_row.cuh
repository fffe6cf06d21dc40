// Row and column kernels of one stage (arXiv:1011.3582; the stage is
// described at the top of engine_impl.cuh) for any of the lengths
// {16, 32, 64, ..., 1024} and {24, 48, ..., 768} of half rows, in fp32 and
// fp64: k1_row, k3_row, k5_row, and the column passes kcol_reg (lengths 16 ..
// 2048 and 24 .. 1536) and kcol_line (4, 6, 8, 12).
//
// What bounds them.  A small grid has few rows: with one block per row
// (kernels_pipe.cuh, kernels_wr.cuh) most SMs idle while a few run long serial
// chains (64^2 fp64: 64 blocks, 88 us for the forward rows).  fp64 is bound by
// the FP64 pipe at any size (two lanes a clock and SM), so its work must be
// spread over all SMs in units smaller than a row.  So here a row is shared by
// a thread-block cluster of CS blocks: each takes 32 / CS of the distribution
// rows (or its share of the derivative rows), and what a site needs from all
// of them (partial moments, derivatives, coefficients) is exchanged through
// distributed shared memory, every block taking a slice of the sites.  No
// block is persistent: the overlap of one row's loads with another's
// transforms comes from several resident blocks per SM.
//
// A half row of H = E P complex values is transformed by P lanes of one warp
// as in kernels_wr.cuh (E-point DFTs, twiddles, one swizzled transpose in
// the row's own buffer, P-point DFTs), generalised: E need not be a multiple
// of P (lane j takes the P-point DFTs k1 = j, j + P, ... < E), rows are padded
// in shared memory so that the row groups of one memory phase use different
// banks, and the tables come from global memory through L1 (a table of its
// own in each short-lived block's shared memory would be a tenth of its
// traffic).  Inverse rows form the packed half-length spectrum straight from
// global memory, with no staging copy.
#pragma once

#include <cooperative_groups.h>

#include "async_copy.cuh"
#include "fft_small.cuh"
#include "row_kernels.h"
#include "stage_layout.cuh"

namespace fftlb {

namespace rk {

namespace cg = cooperative_groups;

// row configuration (see row_p in row_kernels.h)
template <typename real, int H> struct Row {
    using C = typename cplx_of<real>::type;
    static constexpr int P = row_p(H), E = H / P;
    static constexpr int NT = row_nt(sizeof(real), H), NG = NT / P;   // threads, row groups
    static constexpr int CS = row_cs(sizeof(real), H);                // blocks per row
    static constexpr int CHN = 32 / CS;                               // distribution rows per block
    static constexpr int RC = row_stride(sizeof(real), H);            // complex values between rows
    static constexpr int NX = 2 * H;
    static constexpr int NXS = NX / CS;                               // sites per block in the pointwise parts
};

// resident blocks per SM the register allocation allows for: 128 registers a
// thread, fp64 168 (255 for the 24-point first stage)
template <typename real, int H> constexpr int row_minb() {
    return Row<real, H>::NT >= 256 ? 2 : sizeof(real) == 4 ? 4 : Row<real, H>::E >= 24 ? 2 : 3;
}

template <int P> __device__ __forceinline__ unsigned lanes_of_row() {
    if constexpr (P >= 32) return 0xffffffffu;
    else return ((1u << P) - 1u) << ((threadIdx.x & 31) & ~(P - 1));
}

template <typename T> __device__ __forceinline__ T ldro(const T *p) { return __ldg(p); }

// Position of stage-1 output (l, k1) in the row buffer.
template <int P> __device__ __forceinline__ int tp(int l, int k1) { return k1 * P + (l ^ (k1 & (P - 1))); }

// In-place DFT (DIR = -1) or unnormalised inverse (+1) of the H values at z
// by lane j of the row's P lanes; tw[k1 P + l] = exp(-2 pi i l k1 / H).
template <int H, int DIR, typename C>
__device__ __forceinline__ void row_fft(C *z, const C *__restrict__ tw, int j) {
    using real = decltype(z[0].x);
    constexpr int P = Row<real, H>::P, E = Row<real, H>::E;
    const unsigned gm = lanes_of_row<P>();
    C v[E];
#pragma unroll
    for (int t = 0; t < E; ++t) v[t] = z[j + P * t];
    SmallDFT<E, DIR, C>::run(v);
#pragma unroll
    for (int k1 = 1; k1 < E; ++k1) {
        C w = ldro(tw + k1 * P + j);
        if (DIR > 0) w.y = -w.y;
        v[k1] = cmul(v[k1], w);
    }
    __syncwarp(gm);
#pragma unroll
    for (int k1 = 0; k1 < E; ++k1) z[tp<P>(j, k1)] = v[k1];
    __syncwarp(gm);
    if constexpr (P == 2 * E && E == 16) {
        // lane k1 + 16 g: the even (g = 0) or odd l, then one radix-2 step
        // across lane ^ 16 (as row_fft_wr)
        const int k1 = j & 15, g = j >> 4;
        C u[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) u[m] = z[tp<P>(g + 2 * m, k1)];
        SmallDFT<16, DIR, C>::run(u);
        C a[8], b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const C send = g ? u[i] : u[8 + i];
            C recv;
            recv.x = __shfl_xor_sync(0xffffffffu, send.x, 16);
            recv.y = __shfl_xor_sync(0xffffffffu, send.y, 16);
            a[i] = g ? recv : u[i];
            b[i] = g ? u[8 + i] : recv;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            real c, s;
            w32<DIR, real>(i, c, s);
            C t = i == 0 ? b[i] : C{b[i].x * c - b[i].y * s, b[i].x * s + b[i].y * c};
            const C r = DIR < 0 ? cmul_mi(t) : cmul_i(t);   // W_32^8
            t = g ? r : t;
            const int k2 = 8 * g + i;
            z[k1 + 16 * k2] = cadd(a[i], t);
            z[k1 + 16 * (k2 + 16)] = csub(a[i], t);
        }
    } else {
        constexpr int NQ = (E + P - 1) / P;
        C u[NQ][P];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int k1 = j + P * q;
            if (E % P == 0 || k1 < E) {
#pragma unroll
                for (int l = 0; l < P; ++l) u[q][l] = z[tp<P>(l, k1)];
                SmallDFT<P, DIR, C>::run(u[q]);
            }
        }
        __syncwarp(gm);   // every lane's reads are done
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int k1 = j + P * q;
            if (E % P == 0 || k1 < E) {
#pragma unroll
                for (int k2 = 0; k2 < P; ++k2) z[k1 + E * k2] = u[q][k2];
            }
        }
    }
    __syncwarp(gm);
}

// Half-length transform Z of a packed real row -> its one-sided spectrum
// X[0 .. H-1] (real Nyquist value in the imaginary part of X[0]), each bin
// handed to put(k, X[k]).  With s = Z[k] + conj Z[H-k], d = Z[k] - conj
// Z[H-k]: X[k] = s/2 + w, X[H-k] = conj(s/2 - w), w = -i/2 exp(-2 pi i k / 2H)
// d; wh[k] = exp(-2 pi i k / 2H) / 2.
template <int H, typename C, typename Put>
__device__ __forceinline__ void row_post(const C *z, const C *__restrict__ wh, int j, const Put &put) {
    using R = decltype(z[0].x);
    constexpr int P = Row<R, H>::P;
#pragma unroll
    for (int k0 = 0; k0 <= H / 2; k0 += P) {
        const int k = k0 + j;
        if (k > H / 2) break;
        if (k == 0) {
            const C z0 = z[0];
            put(0, C{z0.x + z0.y, z0.x - z0.y});
        } else {
            const C p = z[k], q = z[H - k];
            const C s = cadd(p, cconj(q)), d = csub(p, cconj(q));
            const C w = cmul(ldro(wh + k), cmul_mi(d));
            put(k, C{R(0.5) * s.x + w.x, R(0.5) * s.y + w.y});
            if (H - k != k) put(H - k, C{R(0.5) * s.x - w.x, -(R(0.5) * s.y - w.y)});
        }
    }
}

// One-sided spectrum get(k), k < H -> the packed half-length spectrum Z in z
// (Z[k] = a + i d conj(w), Z[H-k] = conj(a - i d conj(w)), a = X[k] + conj
// X[H-k], d = X[k] - conj X[H-k], w = exp(-2 pi i k / 2H)); U pairs of loads in
// flight.
template <int H, typename C, typename Get>
__device__ __forceinline__ void row_pre(C *z, const C *__restrict__ wp, int j, const Get &get) {
    using R = decltype(z[0].x);
    constexpr int P = Row<R, H>::P, NK = H / (2 * P);   // k = j + P i, i < NK, and k = H / 2
    constexpr int UM = sizeof(R) == 8 ? 4 : 8;
    constexpr int U = NK <= UM ? NK : NK % UM == 0 ? UM : NK % 6 == 0 ? (UM == 8 ? 6 : 3) : 1;
    static_assert(H % (2 * P) == 0, "row configuration");
#pragma unroll 1
    for (int i0 = 0; i0 < NK; i0 += U) {
        C p[U], q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = j + P * (i0 + u);
            p[u] = get(k);
            q[u] = get(k == 0 ? H / 2 : H - k);   // (lane 0's first pair: bins 0 and H / 2)
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = j + P * (i0 + u);
            if (k == 0) {
                z[0] = C{p[u].x + p[u].y, p[u].x - p[u].y};
                // k = H / 2: a = 2 Re X, d = 2 i Im X, i d conj(w) = -2 i Im X
                // with w = -i: Z = 2 conj X
                z[H / 2] = C{R(2) * q[u].x, R(-2) * q[u].y};
            } else {
                const C a = cadd(p[u], cconj(q[u])), d = csub(p[u], cconj(q[u]));
                const C t = cmul_i(cmul(d, cconj(ldro(wp + k))));
                z[k] = cadd(a, t);
                z[H - k] = cconj(csub(a, t));
            }
        }
    }
}

// weight F_k (Eq. 4), k = 0..3: see weight_Fk in engine_impl.cuh
__device__ __forceinline__ double wk(const RowArgs<double> &A, int k, double T) {
    return T * (A.Fk[k][3] + T * (A.Fk[k][2] + T * (A.Fk[k][1] + T * A.Fk[k][0])));
}
__device__ __forceinline__ float wk(const RowArgs<float> &A, int k, float T) {
    float s = A.Fk[k][0], c = A.Fkl[k][0];
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        const float p = __fmul_rn(s, T), pe = fmaf(s, T, -p);
        const float a = A.Fk[k][j];
        const float sn = __fadd_rn(p, a), z = __fsub_rn(sn, p);
        const float se = __fadd_rn(__fsub_rn(p, __fsub_rn(sn, z)), __fsub_rn(a, z));
        c = fmaf(c, T, pe + se + A.Fkl[k][j]);
        s = sn;
    }
    return T * (s + c);
}

template <int CS> __device__ __forceinline__ int block_rank() {
    if constexpr (CS == 1) return 0;
    else return (int)cg::this_cluster().block_rank();
}
// barrier of the row's blocks (their shared memory written so far is visible
// to each other after it)
template <int CS> __device__ __forceinline__ void row_arrive() {
    if constexpr (CS > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
template <int CS> __device__ __forceinline__ void row_wait() {
    if constexpr (CS > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    else __syncthreads();
}
// p's counterpart in block r of the cluster
template <int CS, typename T> __device__ __forceinline__ T *in_block(T *p, int r) {
    if constexpr (CS == 1) return p;
    else return cg::this_cluster().map_shared_rank(p, r);
}

// ---------------------------------------------------------------------------
// K1: moments rho, u, T (Eqs. 7-9), Pi = P^w - rho T (Eq. 18), g = M/T, and the
// forward rows of the 32 moving f_i and of rho, u_x, u_y, T, Pi, g.  Block c of
// the row takes f_i, i = 1 + c CHN ..: it sums their share of the moments,
// transforms them while the other blocks' sums arrive, forms the fields of
// its slice of sites and sends each to the block that transforms it.
// ---------------------------------------------------------------------------

template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) k1_row(const __grid_constant__ RowArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int CS = G::CS, CHN = G::CHN, RC = G::RC, NX = G::NX, NT = G::NT, P = G::P, NXS = G::NXS;
    constexpr int NF = (6 + CS - 1) / CS;   // field rows per block
    extern __shared__ __align__(128) unsigned char row_smem[];
    __shared__ __align__(8) uint64_t bar;
    C *B = reinterpret_cast<C *>(row_smem);                       // [CHN + 1] rows
    C *F = B + (CHN + 1) * RC;                                    // [NF] field rows
    real *pm = reinterpret_cast<real *>(F + NF * RC);             // [4][NX] partial moments
    const int tid = threadIdx.x, c = block_rank<CS>(), j = tid & (P - 1), grp = tid / P;
    const int ny = A.ny, yg = (int)blockIdx.x / CS, run = yg / ny, y = yg - run * ny;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    const real *f = A.f + (size_t)run * Q * N + (size_t)y * NX;
    C *spec = A.spec + (size_t)run * NSLOT * slot + (size_t)y * H;
    const int nrow = c == 0 ? CHN + 1 : CHN;                      // block 0 also sums the rest velocity
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    if (tid == 0) {
        mbar_expect_tx(&bar, (uint32_t)(nrow * NX * sizeof(real)));
        for (int r = 0; r < CHN; ++r)
            bulk_g2s(B + r * RC, f + (size_t)(1 + c * CHN + r) * N, NX * sizeof(real), &bar);
        if (c == 0) bulk_g2s(B + CHN * RC, f, NX * sizeof(real), &bar);
    }
    // (a wait that runs out is recorded and the row carries on: leaving early
    // would pull this block's shared memory from under the others)
    if (!block_wait(&bar, 0, A.err)) mbar_wait_bounded(&bar, 0);
    for (int x = tid; x < NX; x += NT) {
        real m0 = 0, m1 = 0, m2 = 0, m3 = 0;
        if (c == 0) m0 = reinterpret_cast<const real *>(B + CHN * RC)[x];
#pragma unroll 8
        for (int r = 0; r < CHN; ++r) {
            const int i = 1 + c * CHN + r;
            const real v = reinterpret_cast<const real *>(B + r * RC)[x];
            m0 += v;
            m1 += A.vx[i] * v;
            m2 += A.vy[i] * v;
            m3 += A.v2[i] * v;
        }
        pm[x] = m0;
        pm[NX + x] = m1;
        pm[2 * NX + x] = m2;
        pm[3 * NX + x] = m3;
    }
    row_arrive<CS>();
    __syncthreads();
#pragma unroll 1
    for (int r = grp; r < CHN; r += G::NG) {
        const int i = 1 + c * CHN + r;
        C *z = B + r * RC;
        row_fft<H, -1>(z, A.tw, j);
        C *dst = spec + (size_t)(i - 1) * slot;
        if (A.vy[i] == real(0)) {   // i v_x k_x f^ / nx, no column pass
            const real sx = A.vx[i] * A.scale_x;
            row_post<H>(z, A.wh, j, [&](int k, C X) {
                const real m = ldro(A.kx + k) * sx;
                dst[k] = C{-m * X.y, m * X.x};
            });
        } else {
            row_post<H>(z, A.wh, j, [&](int k, C X) { dst[k] = X; });
        }
    }
    row_wait<CS>();
    real *fields = A.fields + (size_t)run * 4 * N + (size_t)y * NX;
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        real m0 = 0, m1 = 0, m2 = 0, m3 = 0;
#pragma unroll
        for (int b = 0; b < CS; ++b) {
            const real *q = in_block<CS>(pm, b);
            m0 += q[x];
            m1 += q[NX + x];
            m2 += q[2 * NX + x];
            m3 += q[3 * NX + x];
        }
        const real rho = m0, ux = m1 / m0, uy = m2 / m0;
        const real T = real(0.5) * (m3 / m0 - (ux * ux + uy * uy));
        fields[x] = rho;
        fields[N + x] = ux;
        fields[2 * N + x] = uy;
        fields[3 * N + x] = T;
        const real lv[6] = {rho, ux, uy, T, rho * T / (real(1) - A.b * rho) - A.a * rho * rho - rho * T,   // Eq. 18
                            (A.K + A.H * T) / T};                                                          // M / T
#pragma unroll
        for (int r = 0; r < 6; ++r) reinterpret_cast<real *>(in_block<CS>(F + (r / CS) * RC, r % CS))[x] = lv[r];
    }
    row_arrive<CS>();
    row_wait<CS>();
    for (int r = c + CS * grp; r < 6; r += CS * G::NG) {
        C *z = F + (r / CS) * RC;
        row_fft<H, -1>(z, A.tw, j);
        C *dst = spec + (size_t)(SLOT_RHO + r) * slot;
        row_post<H>(z, A.wh, j, [&](int k, C X) { dst[k] = X; });
    }
}

template <typename real, int H> size_t k1_row_smem() {
    using G = Row<real, H>;
    return (size_t)(G::CHN + 1 + (6 + G::CS - 1) / G::CS) * G::RC * 2 * sizeof(real) + (size_t)4 * G::NX * sizeof(real);
}

// ---------------------------------------------------------------------------
// K3: inverse rows of the 15 level-1 derivatives (those with a factor k_x
// formed here from the row spectra, stage_layout.cuh) -> Lambda (Eq. 19),
// Phi = 2 q rho T grad T (Eq. 23), the numerators of C (Eq. 22) and B (Eq. 21)
// -> forward rows of Lambda_xx, Lambda_xy, Lambda_yy, Phi_x, Phi_y.  Block c of
// the row transforms the derivative rows o = c, c + CS, ..., takes its slice
// of the sites, and transforms the output rows r = c, c + CS, ....
// ---------------------------------------------------------------------------

template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) k3_row(const __grid_constant__ RowArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int CS = G::CS, RC = G::RC, NX = G::NX, NT = G::NT, P = G::P, NXS = G::NXS;
    constexpr int ND = (ND1 + CS - 1) / CS, NL = (5 + CS - 1) / CS;
    extern __shared__ __align__(128) unsigned char row_smem[];
    C *D = reinterpret_cast<C *>(row_smem);   // [ND] derivative rows
    C *L = D + ND * RC;                       // [NL] output rows
    const int tid = threadIdx.x, c = block_rank<CS>(), j = tid & (P - 1), grp = tid / P;
    const int ny = A.ny, yg = (int)blockIdx.x / CS, run = yg / ny, y = yg - run * ny;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    C *spec = A.spec + (size_t)run * NSLOT * slot + (size_t)y * H;
    const real sx = A.scale_x;
    const real *__restrict__ kx = A.kx;
#pragma unroll 1
    for (int o = c + CS * grp; o < ND1; o += CS * G::NG) {
        C *z = D + (o / CS) * RC;
        // (none of the slots read here is written by this launch)
        const C *__restrict__ s0 = spec + (size_t)(o == D_DIVX ? SLOT_UX : k3_src_slot(o)) * slot;
        if (o == D_LAP) {   // (d_xx + d_yy) rho
            const C *__restrict__ s1 = spec + (size_t)SLOT_RHO * slot;
            row_pre<H>(z, A.wp, j, [&](int k) {
                const C a = ldro(s0 + k), b = ldro(s1 + k);
                const real ax = ldro(kx + k), m = ax * sx;
                return C{a.x - ax * m * b.x, a.y - ax * m * b.y};
            });
        } else if (o == D_DIVX) {   // d_x (d_x u_x + d_y u_y)
            const C *__restrict__ s1 = spec + (size_t)(SLOT_D1 + D_UYY) * slot;
            row_pre<H>(z, A.wp, j, [&](int k) {
                const C a = ldro(s0 + k), b = ldro(s1 + k);
                const real ax = ldro(kx + k), m = ax * sx;
                const C w = C{b.x - m * a.y, b.y + m * a.x};
                return C{-ax * w.y, ax * w.x};
            });
        } else if (o == D_DIVY) {   // d_yy u_y + d_x (d_y u_x)
            const C *__restrict__ s1 = spec + (size_t)(SLOT_D1 + D_UXY) * slot;
            row_pre<H>(z, A.wp, j, [&](int k) {
                const C a = ldro(s0 + k), b = ldro(s1 + k);
                const real ax = ldro(kx + k);
                return C{a.x - ax * b.y, a.y + ax * b.x};
            });
        } else if (o == D_RX || o == D_UXX || o == D_UYX || o == D_TX || o == D_PIX || o == D_GX) {   // d_x
            row_pre<H>(z, A.wp, j, [&](int k) {
                const C a = ldro(s0 + k);
                const real m = ldro(kx + k) * sx;
                return C{-m * a.y, m * a.x};
            });
        } else {   // d_y, from the column pass
            row_pre<H>(z, A.wp, j, [&](int k) { return ldro(s0 + k); });
        }
        __syncwarp(lanes_of_row<P>());
        row_fft<H, +1>(z, A.tw, j);
    }
    row_arrive<CS>();
    row_wait<CS>();
    const real *fields = A.fields + (size_t)run * 4 * N + (size_t)y * NX;
    real *aux = A.aux + (size_t)run * 3 * N + (size_t)y * NX;
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        const real rho = fields[x], T = fields[3 * N + x];
        real d[ND1];
#pragma unroll
        for (int o = 0; o < ND1; ++o) d[o] = reinterpret_cast<const real *>(in_block<CS>(D + (o / CS) * RC, o % CS))[x];
        const real rx = d[D_RX], ry = d[D_RY], div = d[D_UXX] + d[D_UYY];
        const real M = A.K + A.H * T;
        const real Pi = rho * T / (real(1) - A.b * rho) - A.a * rho * rho - rho * T;
        const real grad2 = rx * rx + ry * ry;
        const real iso = -(rho * T * (rx * d[D_GX] + ry * d[D_GY])) - M * (rho * d[D_LAP] + real(0.5) * grad2);   // Eq. 19
        const real Lxx = M * rx * rx + iso, Lxy = M * rx * ry, Lyy = M * ry * ry + iso;
        const real Ldu = Lxx * d[D_UXX] + Lxy * (d[D_UYX] + d[D_UXY]) + Lyy * d[D_UYY];
        const real Cn = Pi * div + Ldu - A.zeta * div * div + A.a * rho * rho * div +
                        A.K * (real(-0.5) * grad2 * div - rho * (rx * d[D_DIVX] + ry * d[D_DIVY]) -
                               (rx * (d[D_UXX] * rx + d[D_UYX] * ry) + ry * (d[D_UXY] * rx + d[D_UYY] * ry)));   // Eq. 22
        aux[x] = Cn;
        aux[N + x] = d[D_PIX] - A.zeta * d[D_DIVX];   // Eq. 21 without d_b Lambda_ab
        aux[2 * N + x] = d[D_PIY] - A.zeta * d[D_DIVY];
        const real q2 = real(2) * A.q * rho * T;   // Eq. 23
        const real lv[5] = {Lxx, Lxy, Lyy, q2 * d[D_TX], q2 * d[D_TY]};
#pragma unroll
        for (int r = 0; r < 5; ++r) reinterpret_cast<real *>(in_block<CS>(L + (r / CS) * RC, r % CS))[x] = lv[r];
    }
    row_arrive<CS>();
    row_wait<CS>();
    for (int r = c + CS * grp; r < 5; r += CS * G::NG) {
        C *z = L + (r / CS) * RC;
        row_fft<H, -1>(z, A.tw, j);
        C *raw = k3_raw_slot(r) >= 0 ? spec + (size_t)k3_raw_slot(r) * slot : nullptr;
        C *mul = k3_mul_slot(r) >= 0 ? spec + (size_t)k3_mul_slot(r) * slot : nullptr;
        row_post<H>(z, A.wh, j, [&](int k, C X) {
            if (raw) raw[k] = X;
            if (mul) {   // the d_x term of level 2
                const real m = ldro(kx + k) * sx;
                mul[k] = C{-m * X.y, m * X.x};
            }
        });
    }
}

template <typename real, int H> size_t k3_row_smem() {
    using G = Row<real, H>;
    return (size_t)((ND1 + G::CS - 1) / G::CS + (5 + G::CS - 1) / G::CS) * G::RC * 2 * sizeof(real);
}

// ---------------------------------------------------------------------------
// K5: inverse rows of the level-2 divergences and the 32 convection terms ->
// A, B, C, C_q (Eqs. 20-23), f^eq (Eq. 3), I (Eq. 11), BGK and the RK
// combination (Eq. 10).  Block c of the row takes the rings of velocities
// 1 + c CHN .. and the level-2 row c (c < 3; with fewer than 3 blocks, rows
// c, c + CS, ...); the coefficients of its slice of sites go to every block.
// ---------------------------------------------------------------------------

constexpr int NCOEF = 5;   // e0, e1x, e1y, C + C_q, 1 / T

// cos(r pi / 4) a + sin(r pi / 4) b with the diagonal sums given: r a
// compile-time constant; dp = (a + b) / sqrt 2, dm = (b - a) / sqrt 2
template <typename real> __device__ __forceinline__ real ring_dot(int r, real a, real b, real dp, real dm) {
    switch (r & 7) {
        case 0: return a;
        case 1: return dp;
        case 2: return b;
        case 3: return dm;
        case 4: return -a;
        case 5: return -dp;
        case 6: return -b;
        default: return -dm;
    }
}

template <typename real, int V> struct Vec;
template <> struct Vec<float, 2> { using T = float2; };
template <> struct Vec<double, 1> { using T = double; };
template <typename real, int V> __device__ __forceinline__ void ldv(real (&a)[V], const real *p) {
    *reinterpret_cast<typename Vec<real, V>::T *>(a) = *reinterpret_cast<const typename Vec<real, V>::T *>(p);
}
template <typename real, int V> __device__ __forceinline__ void stv(real *p, const real (&a)[V]) {
    *reinterpret_cast<typename Vec<real, V>::T *>(p) = *reinterpret_cast<const typename Vec<real, V>::T *>(a);
}

template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) k5_row(const __grid_constant__ RowArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int CS = G::CS, CHN = G::CHN, RC = G::RC, NX = G::NX, NT = G::NT, P = G::P, NXS = G::NXS;
    constexpr int N2 = (3 + CS - 1) / CS, NRING = CHN / 8;
    constexpr int V = sizeof(real) == 4 ? 2 : 1;   // sites per thread and pass of the epilogue
    static_assert(CHN % 8 == 0, "whole rings per block");
    extern __shared__ __align__(128) unsigned char row_smem[];
    C *B = reinterpret_cast<C *>(row_smem);                 // [CHN] convection rows
    C *S = B + CHN * RC;                                    // [N2] level-2 rows
    real *co = reinterpret_cast<real *>(S + N2 * RC);       // [NCOEF][NX]
    const int tid = threadIdx.x, c = block_rank<CS>(), j = tid & (P - 1), grp = tid / P;
    const int ny = A.ny, yg = (int)blockIdx.x / CS, run = yg / ny, y = yg - run * ny;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    const C *__restrict__ spec = A.spec + (size_t)run * NSLOT * slot + (size_t)y * H;
    const size_t fo = (size_t)run * Q * N + (size_t)y * NX;
    const real *fields = A.fields + (size_t)run * 4 * N + (size_t)y * NX;
    const real *aux = A.aux + (size_t)run * 3 * N + (size_t)y * NX;
    const real dt = A.dt, itau = A.itau, alpha = A.alpha, beta = A.beta;
    const bool with_base = alpha != real(0);
    if (tid < CHN) {   // this block's distribution rows into L2 ahead of the epilogue
        const size_t o = fo + (size_t)(1 + c * CHN + tid) * N;
        bulk_prefetch_l2(A.fcur + o, NX * sizeof(real));
        if (with_base) bulk_prefetch_l2(A.fbase + o, NX * sizeof(real));
    }
    // level-2 rows first: the others wait for them
    for (int r = c + CS * grp; r < 3; r += CS * G::NG) {
        C *z = S + (r / CS) * RC;
        const C *__restrict__ src = spec + (size_t)(SLOT_L2 + (r == 0 ? 0 : r + 1)) * slot;
        row_pre<H>(z, A.wp, j, [&](int k) { return ldro(src + k); });
        __syncwarp(lanes_of_row<P>());
        row_fft<H, +1>(z, A.tw, j);
    }
    row_arrive<CS>();
#pragma unroll 1
    for (int r = grp; r < CHN; r += G::NG) {
        C *z = B + r * RC;
        const C *__restrict__ src = spec + (size_t)(c * CHN + r) * slot;
        row_pre<H>(z, A.wp, j, [&](int k) { return ldro(src + k); });
        __syncwarp(lanes_of_row<P>());
        row_fft<H, +1>(z, A.tw, j);
    }
    row_wait<CS>();
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        const real rho = fields[x], ux = fields[N + x], uy = fields[2 * N + x], T = fields[3 * N + x];
        const real fc = A.fcur[fo + x], fb = with_base ? A.fbase[fo + x] : real(0);
        const real a0 = aux[x], a1 = aux[N + x], a2 = aux[2 * N + x];
        const real dLx = reinterpret_cast<const real *>(in_block<CS>(S, 0))[x];
        const real dLy = reinterpret_cast<const real *>(in_block<CS>(S + (1 / CS) * RC, 1 % CS))[x];
        const real dPh = reinterpret_cast<const real *>(in_block<CS>(S + (2 / CS) * RC, 2 % CS))[x];
        const real rT = rho * T, irT = real(1) / rT, iT = real(1) / T;
        const real Bx = (a1 + dLx) * irT, By = (a2 + dLy) * irT;   // Eq. 21
        const real CC = (a0 + dPh) * (real(0.5) * irT * iT);        // C + C_q, Eqs. 22-23
        const real At = real(-2) * CC * T;                          // Eq. 20
        const real u2 = ux * ux + uy * uy;
        // I = -(A + B.(v-u) + CC |v-u|^2) f^eq = -(e0 + e1.v + CC |v|^2) f^eq
        const real e[NCOEF] = {At - (Bx * ux + By * uy) + CC * u2, Bx - real(2) * CC * ux, By - real(2) * CC * uy, CC, iT};
#pragma unroll
        for (int b = 0; b < CS; ++b) {
            real *q = in_block<CS>(co, b);
#pragma unroll
            for (int i = 0; i < NCOEF; ++i) q[i * NX + x] = e[i];
        }
        // the rest velocity (no convection)
        real F0 = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) F0 += wk(A, k, T);
        F0 = real(1) - real(8) * F0;
        const real qq = real(0.5) * u2 * iT, om = real(1) - qq;
        const real fe = rho * F0 * (om + real(0.5) * qq * qq);
        real fn = beta * (fc + dt * (-(fc - fe) * itau - e[0] * fe));
        if (with_base) fn += alpha * fb;
        A.fout[fo + x] = fn;
    }
    row_arrive<CS>();
    row_wait<CS>();
    // the rings of this block: velocities 1 + 8 k .. 8 + 8 k of Eq. 1, one
    // speed, one weight, the eight directions known at compile time
#pragma unroll 1
    for (int it = tid; it < NRING * (NX / V); it += NT) {
        const int rr = NRING == 1 ? 0 : it / (NX / V), x = (NRING == 1 ? it : it - rr * (NX / V)) * V;
        const int k = c * NRING + rr, v0 = 8 * k;
        const real sk = A.vx[1 + v0], sk2 = A.v2[1 + v0];   // direction 0: v = (s_k, 0)
        const size_t o = fo + (size_t)(1 + v0) * N + x;
        const real *pc = A.fcur + o, *pb = A.fbase + o;
        real *po = A.fout + o;
        real fc[8][V], fb[8][V];   // (all loads before any store: fout may be fcur or fbase)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            ldv<real, V>(fc[r], pc + (size_t)r * N);
            if (with_base) ldv<real, V>(fb[r], pb + (size_t)r * N);
        }
        real rho[V], ux[V], uy[V], T[V], e0[V], ex[V], ey[V], CC[V], iT[V];
        ldv<real, V>(rho, fields + x);
        ldv<real, V>(ux, fields + N + x);
        ldv<real, V>(uy, fields + 2 * N + x);
        ldv<real, V>(T, fields + 3 * N + x);
        ldv<real, V>(e0, co + x);
        ldv<real, V>(ex, co + NX + x);
        ldv<real, V>(ey, co + 2 * NX + x);
        ldv<real, V>(CC, co + 3 * NX + x);
        ldv<real, V>(iT, co + 4 * NX + x);
        const real hh = real(0.70710678118654752440);
        real p0[V], p1[V], p2[V], p3[V], p4[V], g0[V], dp[V], dm[V], ep[V], em[V];
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const real qq = real(0.5) * (ux[q] * ux[q] + uy[q] * uy[q]) * iT[q], om = real(1) - qq;
            const real rF = rho[q] * wk(A, k, T[q]);   // Eq. 4
            const real r1 = rF * iT[q], r2 = r1 * iT[q], r3 = r2 * iT[q];
            p0[q] = rF * (om + real(0.5) * qq * qq);   // rho F_k times the factors of Eq. 3
            p1[q] = r1 * om;
            p2[q] = real(0.5) * r2 * om;
            p3[q] = r3 * (real(1) / real(6));
            p4[q] = r3 * iT[q] * (real(1) / real(24));
            g0[q] = e0[q] + CC[q] * sk2;
            ux[q] *= sk;
            uy[q] *= sk;
            ex[q] *= sk;
            ey[q] *= sk;
            dp[q] = hh * (ux[q] + uy[q]);
            dm[q] = hh * (uy[q] - ux[q]);
            ep[q] = hh * (ex[q] + ey[q]);
            em[q] = hh * (ey[q] - ex[q]);
        }
        const real *cr = reinterpret_cast<const real *>(B + rr * 8 * RC) + x;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            real cv[V], fn[V];
            ldv<real, V>(cv, cr + (size_t)r * 2 * RC);
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const real vu = ring_dot<real>(r, ux[q], uy[q], dp[q], dm[q]);
                const real fe = p0[q] + vu * (p1[q] + vu * (p2[q] + vu * (p3[q] + vu * p4[q])));   // Eq. 3
                const real g = g0[q] + ring_dot<real>(r, ex[q], ey[q], ep[q], em[q]);             // -I / f^eq, Eq. 11
                const real rhs = -cv[q] - (fc[r][q] - fe) * itau - g * fe;                          // Eq. 10
                fn[q] = beta * (fc[r][q] + dt * rhs);
                if (with_base) fn[q] += alpha * fb[r][q];
            }
            stv<real, V>(po + (size_t)r * N, fn);
        }
    }
}

template <typename real, int H> size_t k5_row_smem() {
    using G = Row<real, H>;
    return (size_t)(G::CHN + (3 + G::CS - 1) / G::CS) * G::RC * 2 * sizeof(real) + (size_t)NCOEF * G::NX * sizeof(real);
}

template <typename real, int H> RowSet row_set() {
    using G = Row<real, H>;
    RowSet s;
    s.k1 = (const void *)&k1_row<real, H>;
    s.k3 = (const void *)&k3_row<real, H>;
    s.k5 = (const void *)&k5_row<real, H>;
    s.nt = G::NT;
    s.cs = G::CS;
    s.smem1 = k1_row_smem<real, H>();
    s.smem3 = k3_row_smem<real, H>();
    s.smem5 = k5_row_smem<real, H>();
    return s;
}

}  // namespace rk

}  // namespace fftlb

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
// of them (partial moments, derivatives, coefficients) goes through distributed
// shared memory, every block taking a slice of the sites.  No block is
// persistent: the overlap of one row's loads with another's
// transforms comes from several resident blocks per SM.
//
// A half row of H = E P complex values is transformed by P lanes of one warp
// as in kernels_wr.cuh (E-point DFTs, twiddles, one swizzled transpose in
// the row's own buffer, P-point DFTs), generalised: E need not be a multiple
// of P (lane j takes the P-point DFTs k1 = j, j + P, ... < E), rows are padded
// in shared memory so that the row groups of one memory phase use different
// banks, and the tables come by one bulk copy that overlaps the first loads
// (through L1 they are cold in every launch).  Inverse rows form the packed
// half-length spectrum straight from global memory, with no staging copy.
//
// The stage's kernels are launched with programmatic stream serialization and
// no explicit trigger: a launch's blocks start as the one before ends, without
// the full hand-over between grids, and wait for its memory (grid_dep_wait) once
// their barriers and tables are under way and before they touch anything the
// stage writes.  A step on 64^2 fp32 83 -> 50 us, on 64^2 fp64 241 -> 204, on
// 2048^2 fp32 4618 -> 4547.  Triggered early instead, the waiting blocks fill the
// SMs that are idle first and then run crowded there (64^2 fp64 389 us).
// What the stage writes is read by ordinary loads: read-only ones are for memory
// that nothing writes while the kernel runs, and these kernels run from before
// their wait on.
#pragma once

#include <cooperative_groups.h>

#include "async_copy.cuh"
#include "block_sum.cuh"
#include "col_kernels.h"
#include "fft_small.cuh"
#include "row_kernels.h"
#include "stage_layout.cuh"
#include "stage_site.cuh"

namespace fftlb {

namespace rk {

namespace cg = cooperative_groups;

// row configuration (see row_p in row_kernels.h)
template <typename real, int H, int NT_ = row_nt((int)sizeof(real), H)> struct Row {
    using C = typename cplx_of<real>::type;
    static constexpr int P = row_p((int)sizeof(real), H), E = H / P;
    static constexpr int NT = NT_, NG = NT / P;                       // threads, row groups
    static constexpr int CS = row_cs((int)sizeof(real), H);           // blocks per row
    static constexpr int CHN = 32 / CS;                               // distribution rows per block
    static constexpr int RC = row_stride((int)sizeof(real), H);            // complex values between rows
    static constexpr int NX = 2 * H;
    static constexpr int NXS = NX / CS;                               // sites per block in the pointwise parts
    static constexpr int NRING = CHN / 8;                             // rings of velocities per block
    // n rows shared by the blocks, in units of the rows of one warp (a warp
    // with one row takes as long as a full one, which is what counts in fp64):
    // row r belongs to block owner(r), as its row local(r) < share(n)
    static constexpr int RPW = 32 / P;
    static __host__ __device__ constexpr int owner(int r) { return (r / RPW) % CS; }
    static __host__ __device__ constexpr int local(int r) { return r / (RPW * CS) * RPW + r % RPW; }
    static __host__ __device__ constexpr int share(int n) { return (n + RPW * CS - 1) / (RPW * CS) * RPW; }
    // block c's rows among n
    static __host__ __device__ constexpr int nrows(int c, int n) {
        int m = 0;
        for (int r = 0; r < n; ++r) m += owner(r) == c;
        return m;
    }
    // the i-th row of block c
    static __host__ __device__ constexpr int nth(int c, int i) { return (i / RPW * CS + c) * RPW + i % RPW; }
};

// resident blocks per SM the register allocation allows for: 128 registers a
// thread, 255 for the 24-point first stage in fp64 (168 for all of fp64 was one
// wave more for K3 on 256^2: 128 us against 95)
template <typename real, int H> constexpr int row_minb() {
    return Row<real, H>::NT >= 256 ? 2 : sizeof(real) == 4 ? 4 : Row<real, H>::E >= 24 ? 2 : 4;
}

template <typename real, int H> constexpr int row_minb3() {
    return row_minb<real, H>() * (Row<real, H>::NT / row_nt3((int)sizeof(real), H));
}

template <int P> __device__ __forceinline__ unsigned lanes_of_row() {
    if constexpr (P >= 32) return 0xffffffffu;
    else return ((1u << P) - 1u) << ((threadIdx.x & 31) & ~(P - 1));
}

// The table block [wh][kx][tw][wp] (row_table): K1 takes its first three
// parts, K5 the last two, K3 all.
template <typename real, int H> struct Tab {
    using C = typename cplx_of<real>::type;
    using L = RowTable<real>;
    const C *wh, *tw, *wp;
    const real *kx;
    // in shared memory at p, holding the parts from byte `from` on
    __device__ __forceinline__ Tab(const unsigned char *p, unsigned from)
        : wh(reinterpret_cast<const C *>(p - from)), tw(reinterpret_cast<const C *>(p + L::tw(H) - from)),
          wp(reinterpret_cast<const C *>(p + L::wp(H) - from)), kx(reinterpret_cast<const real *>(p + L::kx(H) - from)) {}
};
// thread 0: barrier, then the copy of bytes [from, to) of the block to dst
template <typename C>
__device__ __forceinline__ void table_issue(unsigned char *dst, const C *tab, unsigned from, unsigned to, uint64_t *bar) {
    bulk_g2s(dst, reinterpret_cast<const unsigned char *>(tab) + from, to - from, bar);
}

// Position of stage-1 output (l, k1) in the row buffer.
template <int P> __device__ __forceinline__ int tp(int l, int k1) { return k1 * P + (l ^ (k1 & (P - 1))); }

// In-place DFT (DIR = -1) or unnormalised inverse (+1) of the H values at z
// by lane j of the row's P lanes; tw[k1 P + l] = exp(-2 pi i l k1 / H).
template <int H, int DIR, typename C>
__device__ __forceinline__ void row_fft(C *z, const C *tw, int j) {
    using real = decltype(z[0].x);
    constexpr int P = Row<real, H>::P, E = Row<real, H>::E;
    const unsigned gm = lanes_of_row<P>();
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
__device__ __forceinline__ void row_post(const C *z, const C *wh, int j, const Put &put) {
    using R = decltype(z[0].x);
    constexpr int P = Row<R, H>::P;
    static_assert(H % (2 * P) == 0, "row configuration");
#pragma unroll
    for (int k0 = 0; k0 < H / 2; k0 += P) {
        const int k = k0 + j;
        if (k == 0) {   // bins 0 and H / 2
            const C z0 = z[0];
            put(0, C{z0.x + z0.y, z0.x - z0.y});
            put(H / 2, cconj(z[H / 2]));
        } else {
            const C p = z[k], q = z[H - k];
            const C s = cadd(p, cconj(q)), d = csub(p, cconj(q));
            const C w = cmul(wh[k], cmul_mi(d));
            put(k, C{R(0.5) * s.x + w.x, R(0.5) * s.y + w.y});
            put(H - k, C{R(0.5) * s.x - w.x, -(R(0.5) * s.y - w.y)});
        }
    }
}

// One-sided spectrum X[k] = form(k, a[k], b[k]), k < H, from the global rows a
// (and b, NS = 2) -> the packed half-length spectrum Z in z (Z[k] = t + i d
// conj(w), Z[H-k] = conj(t - i d conj(w)), t = X[k] + conj X[H-k], d = X[k] - conj
// X[H-k], w = exp(-2 pi i k / 2H)); U pairs of loads in flight, ready() between
// the first ones and their use.
template <int H, int NS, typename C, typename Form, typename Ready>
__device__ __forceinline__ void row_pre(C *z, const C *wp, int j, const C *__restrict__ a, const C *__restrict__ b,
                                        const Form &form, const Ready &ready) {
    using R = decltype(z[0].x);
    constexpr int P = Row<R, H>::P, NK = H / (2 * P);   // k = j + P i, i < NK, and k = H / 2
    constexpr int UM = sizeof(R) == 8 ? 4 : 8;
    constexpr int U = NK <= UM ? NK : NK % UM == 0 ? UM : NK % 6 == 0 ? (UM == 8 ? 6 : 3) : 1;
    static_assert(H % (2 * P) == 0, "row configuration");
#pragma unroll 1
    for (int i0 = 0; i0 < NK; i0 += U) {
        C pa[U], qa[U], pb[NS > 1 ? U : 1], qb[NS > 1 ? U : 1];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = j + P * (i0 + u), kc = k == 0 ? H / 2 : H - k;   // (lane 0's first pair: bins 0 and H / 2)
            pa[u] = a[k];
            qa[u] = a[kc];
            if constexpr (NS > 1) {
                pb[u] = b[k];
                qb[u] = b[kc];
            }
        }
        if (i0 == 0) ready();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = j + P * (i0 + u), kc = k == 0 ? H / 2 : H - k;
            const C p = form(k, pa[u], pb[NS > 1 ? u : 0]), q = form(kc, qa[u], qb[NS > 1 ? u : 0]);
            if (k == 0) {
                z[0] = C{p.x + p.y, p.x - p.y};
                // k = H / 2: t = 2 Re X, d = 2 i Im X, i d conj(w) = -2 i Im X
                // with w = -i: Z = 2 conj X
                z[H / 2] = C{R(2) * q.x, R(-2) * q.y};
            } else {
                const C t = cadd(p, cconj(q)), d = csub(p, cconj(q));
                const C e = cmul_i(cmul(d, cconj(wp[k])));
                z[k] = cadd(t, e);
                z[H - k] = cconj(csub(t, e));
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

// this thread's bounded wait for the tables or (PEER) for what the row's other
// blocks push; running out is recorded
template <bool PEER = false> __device__ __forceinline__ void table_wait(uint64_t *bar, int *err) {
    if (!mbar_wait_bounded<PEER>(bar, 0)) {
        atomicOr(err, kErrWaitTimeout);
        mbar_wait_bounded<PEER>(bar, 0);
    }
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
// The row's blocks push what each other needs instead of reading it behind a
// barrier: copies and stores into another block's shared memory that complete on
// that block's mbarrier need no fence, while a cluster barrier's release holds
// every warp until all its accesses have been performed.  A block stays until
// the others are done with its memory: row_leave() where it needs nothing more
// from them, row_gone() at its end (no data is handed over by these two).
// Against a cluster barrier for every hand-over: 384^2 fp32 215 -> 196 us a step,
// 768^2 699 -> 650, 2048^2 4480 -> 4288 (K5 562 -> 521), 128^2 64.2 -> 60.4, 64^2
// fp64 204 -> 198.  The first hand-over of K1 and K3 keeps the barrier: pushed,
// it needs room for three more rows, a resident block less on the long ones, and
// one release a block on the others' mbarriers took as long (384^2: 198).
template <int CS> __device__ __forceinline__ void row_leave() {
    if constexpr (CS > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
}
template <int CS> __device__ __forceinline__ void row_gone() {
    if constexpr (CS > 1) asm volatile("barrier.cluster.wait;" ::: "memory");
}
// p's address in block r's part of the cluster's shared memory
__device__ __forceinline__ uint32_t peer_u32(const void *p, int r) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(r));
    return a;
}
// v to p in block r, completing on bar in block r
__device__ __forceinline__ void push(float *p, float v, uint64_t *bar, int r) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(peer_u32(p, r)),
                 "r"(__float_as_uint(v)), "r"(peer_u32(bar, r))
                 : "memory");
}
__device__ __forceinline__ void push(double *p, double v, uint64_t *bar, int r) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(peer_u32(p, r)),
                 "l"(__double_as_longlong(v)), "r"(peer_u32(bar, r))
                 : "memory");
}
// `bytes` (a multiple of 16, both addresses 16-byte aligned) from src of this
// block to dst in block r, completing on bar in block r
__device__ __forceinline__ void push_bulk(void *dst, const void *src, uint32_t bytes, uint64_t *bar, int r) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     peer_u32(dst, r)),
                 "r"(smem_u32(src)), "r"(bytes), "r"(peer_u32(bar, r))
                 : "memory");
}

// p's counterpart in block r of the cluster
template <int CS, typename T> __device__ __forceinline__ T *in_block(T *p, int r) {
    if constexpr (CS == 1) return p;
    else return cg::this_cluster().map_shared_rank(p, r);
}

// ---------------------------------------------------------------------------
// K1: moments rho, u, T (Eqs. 7-9), Pi = P^w - rho T (Eq. 18), g = M/T, and the
// forward rows of the f_i with v_x != 0 and of rho, u_x, u_y, T, Pi, g.  Block c
// of the row takes f_i, i = 1 + c CHN ..: it sums their share of the moments,
// forms the fields of its slice of sites from everybody's sums, pushes each
// field to the block that transforms it, and then transforms its f_i and its
// share of the fields together (the fields after the f_i, hiding the exchange,
// took a second pass of the same length: 51 us against 37 on six 512x4 fp64
// slabs).
// ---------------------------------------------------------------------------

template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) k1_row(const __grid_constant__ RowArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int CS = G::CS, CHN = G::CHN, RC = G::RC, NX = G::NX, NT = G::NT, P = G::P, NXS = G::NXS, NR = G::NRING;
    extern __shared__ __align__(128) unsigned char row_smem[];
    __shared__ __align__(8) uint64_t bar, fbar;
    using LT = RowTable<real>;
    C *B = reinterpret_cast<C *>(row_smem);     // [CHN + 1] rows
    C *F = B + (CHN + 1) * RC;                  // [share(6)] field rows
    C *S = F + G::share(6) * RC;                // [2 NR - 1] rows: partial moments, see pm
    unsigned char *tb = reinterpret_cast<unsigned char *>(S + (2 * NR - 1) * RC);
    const Tab<real, H> T(tb, 0);
    // partial moment m of ring rr: two take the rows of the ring's directions 2
    // and 6, which no transform needs (each site's values are read and replaced
    // by one thread), one of all the rest velocity's row, the others rows of S
    auto pm = [&](int rr, int m) -> real * {
        C *p = m < 2 ? B + (rr * 8 + 2 + 4 * m) * RC : m == 2 && rr == 0 ? B + CHN * RC : S + (2 * rr + m - 3) * RC;
        return reinterpret_cast<real *>(p);
    };
    const int c = block_rank<CS>(), tid = (int)threadIdx.x, j = tid & (P - 1), grp = tid / P;
    const int ny = A.ny, yg = (int)blockIdx.x / CS, run = yg / ny, y = yg - run * ny;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    const real *f = A.f + (size_t)run * Q * N + (size_t)y * NX;
    C *spec = A.spec + (size_t)run * NSLOT * slot + (size_t)y * H;
    const int nrow = c == 0 ? CHN + 1 : CHN;                      // block 0 also sums the rest velocity
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init(&fbar, 1);
        mbar_init_fence();
        mbar_expect_tx(&fbar, G::nrows(c, 6) * NX * sizeof(real));   // its field rows, from every block
    }
    __syncthreads();
    grid_dep_wait();
    if (tid == 0) {
        mbar_expect_tx(&bar, (uint32_t)(nrow * NX * sizeof(real)) + LT::wp(H));
        for (int r = 0; r < CHN; ++r)
            bulk_g2s(B + r * RC, f + (size_t)(1 + c * CHN + r) * N, NX * sizeof(real), &bar);
        if (c == 0) bulk_g2s(B + CHN * RC, f, NX * sizeof(real), &bar);
        table_issue(tb, A.tab, 0, LT::wp(H), &bar);
    }
    // (a wait that runs out is recorded and the row carries on: leaving early
    // would pull this block's shared memory from under the others)
    if (!block_wait(&bar, 0, A.err)) mbar_wait_bounded(&bar, 0);
    // one ring at one site: speed s, directions r pi / 4 (19 operations instead
    // of 32 with the velocities one by one)
    const real hh = real(0.70710678118654752440);
    for (int it = tid; it < NR * NX; it += NT) {
        const int rr = NR == 1 ? 0 : it / NX, x = NR == 1 ? it : it - rr * NX;
        const int v0 = 1 + c * CHN + 8 * rr;
        const real sk = A.vx[v0], sk2 = A.v2[v0];
        real v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = reinterpret_cast<const real *>(B + (rr * 8 + r) * RC)[x];
        const real d04 = v[0] - v[4], d15 = v[1] - v[5], d26 = v[2] - v[6], d37 = v[3] - v[7];
        const real sum = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
        real m0 = sum;
        if (c == 0 && rr == 0) m0 += reinterpret_cast<const real *>(B + CHN * RC)[x];
        pm(rr, 0)[x] = m0;
        pm(rr, 1)[x] = sk * (d04 + hh * (d15 - d37));
        pm(rr, 2)[x] = sk * (d26 + hh * (d15 + d37));
        pm(rr, 3)[x] = sk2 * sum;
    }
    row_arrive<CS>();
    row_wait<CS>();
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        real m0 = 0, m1 = 0, m2 = 0, m3 = 0;
#pragma unroll
        for (int b = 0; b < CS; ++b) {
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                m0 += in_block<CS>(pm(rr, 0), b)[x];
                m1 += in_block<CS>(pm(rr, 1), b)[x];
                m2 += in_block<CS>(pm(rr, 2), b)[x];
                m3 += in_block<CS>(pm(rr, 3), b)[x];
            }
        }
        const real rho = m0, ux = m1 / m0, uy = m2 / m0;
        const real Te = real(0.5) * (m3 / m0 - (ux * ux + uy * uy));
        const real lv[6] = {rho, ux, uy, Te, rho * Te / (real(1) - A.b * rho) - A.a * rho * rho - rho * Te,   // Eq. 18
                            (A.K + A.H * Te) / Te};                                                        // M / T
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            real *q = reinterpret_cast<real *>(F + G::local(r) * RC) + x;
            if constexpr (CS == 1) *q = lv[r];
            else push(q, lv[r], &fbar, G::owner(r));
        }
    }
    if constexpr (CS == 1) __syncthreads();
    row_leave<CS>();   // (has read the others' sums; its field rows come by fbar)
    // this block's distribution rows and its share of the field rows, one row
    // group each: 6 of every 8 directions leave room for the fields
    static_assert(6 * NR + G::share(6) <= G::NG, "one pass");
    if (grp < 6 * NR) {
        const int rr = NR == 1 ? 0 : grp / 6, r = rr * 8 + ring_dir(grp - 6 * rr), i = 1 + c * CHN + r;
        C *z = B + r * RC;
        row_fft<H, -1>(z, T.tw, j);
        C *dst = spec + (size_t)(i - 1) * slot;
        if (A.vy[i] == real(0)) {   // i v_x k_x f^ / nx, no column pass
            const real sx = A.vx[i] * A.scale_x;
            row_post<H>(z, T.wh, j, [&](int k, C X) {
                const real m = T.kx[k] * sx;
                dst[k] = C{-m * X.y, m * X.x};
            });
        } else {
            row_post<H>(z, T.wh, j, [&](int k, C X) { dst[k] = X; });
        }
    } else {
        const int q = grp - 6 * NR, r = G::nth(c, q);
        if (q < G::share(6) && r < 6) {
            if constexpr (CS > 1) table_wait<true>(&fbar, A.err);
            C *z = F + q * RC;
            C *real_row = spec + (size_t)(SLOT_F + r) * slot, *dst = spec + (size_t)(SLOT_RHO + r) * slot;
#pragma unroll
            for (int k = j; k < H; k += P) real_row[k] = z[k];
            row_fft<H, -1>(z, T.tw, j);
            row_post<H>(z, T.wh, j, [&](int k, C X) { dst[k] = X; });
        }
    }
    row_gone<CS>();
}

template <typename real, int H> size_t k1_row_smem() {
    using G = Row<real, H>;
    return (size_t)(G::CHN + 1 + G::share(6) + 2 * G::NRING - 1) * G::RC * 2 * sizeof(real) + RowTable<real>::wp(H);
}

// ---------------------------------------------------------------------------
// K3: inverse rows of the 11 level-1 derivatives that have a factor k_x or
// start from a row spectrum (stage_layout.cuh) -> Lambda (Eq. 19), Phi (Eq. 23),
// the numerators of C (Eq. 22) and B (Eq. 21) -> the row spectra of d_x of Phi_x,
// Lambda_xx, Lambda_xy.  Their inverse rows are K5's, which has row groups to
// spare for them; here they would be a third pass in a row (68 us against 52
// on six 512x4 fp64 slabs).
// ---------------------------------------------------------------------------

template <typename real, int H>
__global__ void __launch_bounds__(row_nt3((int)sizeof(real), H), row_minb3<real, H>()) k3_row(const __grid_constant__ RowArgs<real> A) {
    using G = Row<real, H, row_nt3((int)sizeof(real), H)>;
    using C = typename G::C;
    constexpr int CS = G::CS, RC = G::RC, NX = G::NX, NT = G::NT, P = G::P, NXS = G::NXS;
    constexpr int ND = G::share(NSP), NL = G::share(3);
    extern __shared__ __align__(128) unsigned char row_smem[];
    C *D = reinterpret_cast<C *>(row_smem);   // [ND] derivative rows
    C *L = D + ND * RC;                       // [NL] Phi_x, Lambda_xx, Lambda_xy
    using LT = RowTable<real>;
    unsigned char *tb = reinterpret_cast<unsigned char *>(L + NL * RC);
    const Tab<real, H> T(tb, 0);
    __shared__ __align__(8) uint64_t bar, lbar;
    const int c = block_rank<CS>(), tid = (int)threadIdx.x, j = tid & (P - 1), grp = tid / P;
    const int ny = A.ny, yg = (int)blockIdx.x / CS, run = yg / ny, y = yg - run * ny;
    const size_t slot = (size_t)ny * H;
    C *spec = A.spec + (size_t)run * NSLOT * slot + (size_t)y * H;
    const real sx = A.scale_x;
    const real *kx = T.kx;
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init(&lbar, 1);
        mbar_init_fence();
        mbar_expect_tx(&lbar, G::nrows(c, 3) * NX * sizeof(real));   // its rows of L, from every block
        mbar_expect_tx(&bar, LT::bytes(H));
        table_issue(tb, A.tab, 0, LT::bytes(H), &bar);
    }
    __syncthreads();
    grid_dep_wait();
    bool first = true;
    auto ready = [&]() {   // the tables are there (a wait that runs out is recorded; see k1_row)
        if (first) table_wait(&bar, A.err);
        first = false;
    };
    // the real rows of this block's slice of sites into L2 (if they are not
    // there) ahead of the pointwise part
    if (tid < NK3 - NSP)
        bulk_prefetch_l2(reinterpret_cast<const real *>(spec + (size_t)k3_src_slot(NSP + tid) * slot) + c * NXS,
                         NXS * sizeof(real));
#pragma unroll 1
    for (int q = grp; q < ND; q += G::NG) {
        const int o = G::nth(c, q);
        if (o >= NSP) continue;
        C *z = D + q * RC;
        // (none of the slots read here is written by this launch)
        const int s = o == D_LAP ? SLOT_RHO : o == D_DIVX ? SLOT_UX : o == D_DIVY ? SLOT_D1 + D1_UXY : k3_src_slot(o);
        const C *__restrict__ s0 = spec + (size_t)s * slot;
        if (o == D_LAP) {   // d_xx rho
            row_pre<H, 1>(z, T.wp, j, s0, s0, [&](int k, C a, C) {
                const real ax = kx[k], m = -ax * (ax * sx);
                return C{m * a.x, m * a.y};
            }, ready);
        } else if (o == D_DIVX) {   // d_x (d_x u_x + d_y u_y)
            row_pre<H, 2>(z, T.wp, j, s0, spec + (size_t)(SLOT_D1 + D1_UYY) * slot, [&](int k, C a, C b) {
                const real ax = kx[k], m = ax * sx;
                const C w = C{b.x - m * a.y, b.y + m * a.x};
                return C{-ax * w.y, ax * w.x};
            }, ready);
        } else if (o == D_UXY || o == D_UYY) {   // d_y, from the column pass
            row_pre<H, 1>(z, T.wp, j, s0, s0, [](int, C a, C) { return a; }, ready);
        } else {   // d_x (of d_y u_x, which carries its 1 / nx, for D_DIVY)
            const real sm = o == D_DIVY ? real(1) : sx;
            row_pre<H, 1>(z, T.wp, j, s0, s0, [&](int k, C a, C) {
                const real m = kx[k] * sm;
                return C{-m * a.y, m * a.x};
            }, ready);
        }
        __syncwarp(lanes_of_row<P>());
        row_fft<H, +1>(z, T.tw, j);
    }
    row_arrive<CS>();
    row_wait<CS>();
    ready();   // (a group without a derivative row has not waited yet)
    auto row = [&](int s) { return reinterpret_cast<real *>(spec + (size_t)s * slot); };
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        real d[NK3];
#pragma unroll
        for (int o = NSP; o < NK3; ++o) d[o] = row(k3_src_slot(o))[x];
#pragma unroll
        for (int o = 0; o < NSP; ++o)
            d[o] = reinterpret_cast<const real *>(in_block<CS>(D + G::local(o) * RC, G::owner(o)))[x];
        const Level2<real> l = level2_site<real>([&](int o) { return d[o]; }, A);
        const real lv[3] = {l.Phx, l.Lxx, l.Lxy};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            real *q = reinterpret_cast<real *>(L + G::local(r) * RC) + x;
            if constexpr (CS == 1) *q = lv[r];
            else push(q, lv[r], &lbar, G::owner(r));
        }
        row(SLOT_A)[x] = l.Cn;
        row(SLOT_A + 1)[x] = l.Bx;
        row(SLOT_A + 2)[x] = l.By;
        row(SLOT_L2)[x] = l.Lxy;
        row(SLOT_L2 + 1)[x] = l.Lyy;
        row(SLOT_L2 + 2)[x] = l.Phy;
    }
    if constexpr (CS == 1) __syncthreads();
    row_leave<CS>();   // (has read the others' rows; its rows of L come by lbar)
    for (int q = grp; q < NL; q += G::NG) {
        const int r = G::nth(c, q);
        if (r >= 3) continue;
        if constexpr (CS > 1) table_wait<true>(&lbar, A.err);
        C *z = L + q * RC;
        row_fft<H, -1>(z, T.tw, j);
        C *dst = spec + (size_t)(SLOT_X + r) * slot;
        row_post<H>(z, T.wh, j, [&](int k, C X) {
            const real m = kx[k] * sx;
            dst[k] = C{-m * X.y, m * X.x};
        });
    }
    row_gone<CS>();
}

template <typename real, int H> size_t k3_row_smem() {
    using G = Row<real, H, row_nt3((int)sizeof(real), H)>;
    return (size_t)(G::share(NSP) + G::share(3)) * G::RC * 2 * sizeof(real) + RowTable<real>::bytes(H);
}

// ---------------------------------------------------------------------------
// K5: inverse rows of the convection terms with v_x != 0 and of the d_x terms of
// level 2, in one pass; A, B, C, C_q (Eqs. 20-23) from the latter, the numerators
// and the column passes of level 2; f^eq (Eq. 3), I (Eq. 11), BGK and the RK
// combination (Eq. 10).  Block c of the row takes the rings of velocities
// 1 + c CHN ..; the coefficients of its slice of sites go to every block.
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
template <> struct Vec<float, 4> { using T = float4; };
template <> struct Vec<double, 1> { using T = double; };
template <typename real, int V> __device__ __forceinline__ void ldv(real (&a)[V], const real *p) {
    *reinterpret_cast<typename Vec<real, V>::T *>(a) = *reinterpret_cast<const typename Vec<real, V>::T *>(p);
}
// f^n of the later Runge-Kutta stages and the new f leave the L2 first: they are
// not read again before the spectra are (2048^2 fp32 592 -> 562 us, 768^2 103.6 ->
// 101.8; the same for K1's reads of f cost 2048^2 326 -> 333, and for the stage
// state gave nothing)
template <typename real, int V> __device__ __forceinline__ void ldv_once(real (&a)[V], const real *p) {
    *reinterpret_cast<typename Vec<real, V>::T *>(a) = __ldcs(reinterpret_cast<const typename Vec<real, V>::T *>(p));
}
template <typename real, int V> __device__ __forceinline__ void stv_once(real *p, const real (&a)[V]) {
    __stcs(reinterpret_cast<typename Vec<real, V>::T *>(p), *reinterpret_cast<const typename Vec<real, V>::T *>(a));
}

template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) k5_row(const __grid_constant__ RowArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int CS = G::CS, CHN = G::CHN, RC = G::RC, NX = G::NX, NT = G::NT, P = G::P, NXS = G::NXS;
    constexpr int NRING = G::NRING;
    // sites per thread and pass of the epilogue, and ring pairs (r, r + 4) loaded
    // before any of their stores: 16-byte accesses on long rows (two halves of a
    // ring, for the registers), all 8 directions at once on short ones
    constexpr int V = sizeof(real) == 8 ? 1 : H >= 256 ? 4 : 2, RP = V == 4 ? 2 : 4;
    static_assert(CHN % 8 == 0, "whole rings per block");
    extern __shared__ __align__(128) unsigned char row_smem[];
    C *B = reinterpret_cast<C *>(row_smem);                     // [6 NRING] convection rows
    C *X = B + 6 * NRING * RC;                                  // [share(3)] d_x rows
    real *co = reinterpret_cast<real *>(X + G::share(3) * RC);  // [NCOEF][NX]
    using LT = RowTable<real>;
    unsigned char *tb = reinterpret_cast<unsigned char *>(co + NCOEF * NX);
    const Tab<real, H> TB(tb, LT::tw(H));
    __shared__ __align__(8) uint64_t bar, xbar, cbar;
    const int c = block_rank<CS>(), tid = (int)threadIdx.x, j = tid & (P - 1), grp = tid / P;
    const int ny = A.ny, yg = (int)blockIdx.x / CS, run = yg / ny, y = yg - run * ny;
    const size_t N = (size_t)NX * ny, slot = (size_t)ny * H;
    const C *__restrict__ spec = A.spec + (size_t)run * NSLOT * slot + (size_t)y * H;
    const size_t fo = (size_t)run * Q * N + (size_t)y * NX;
    auto row = [&](int s) { return reinterpret_cast<const real *>(spec + (size_t)s * slot); };
    const real dt = A.dt, itau = A.itau, beta = A.beta;
    const bool with_base = A.alpha != real(0);
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init(&xbar, 1);
        mbar_init(&cbar, 1);
        mbar_init_fence();
        mbar_expect_tx(&xbar, 3 * NXS * sizeof(real));                  // d_x at this block's slice
        mbar_expect_tx(&cbar, (CS - 1) * NCOEF * NXS * sizeof(real));   // the other slices' coefficients
        mbar_expect_tx(&bar, LT::bytes(H) - LT::tw(H));
        table_issue(tb, A.tab, LT::tw(H), LT::bytes(H), &bar);
    }
    __syncthreads();
    row_leave<CS>();   // (the barriers are initialised)
    grid_dep_wait();
    if (tid < CHN) {   // this block's distribution rows into L2 ahead of the epilogue
        const size_t o = fo + (size_t)(1 + c * CHN + tid) * N;
        bulk_prefetch_l2(A.fcur + o, NX * sizeof(real));
        if (with_base) bulk_prefetch_l2(A.fbase + o, NX * sizeof(real));
    }
    bool first = true;
    auto ready = [&]() {   // the tables are there (a wait that runs out is recorded; see k1_row)
        if (first) table_wait(&bar, A.err);
        first = false;
    };
    static_assert(6 * NRING + G::share(3) <= G::NG, "one pass");
    {
        const int rr = NRING == 1 ? 0 : grp / 6, q = grp - 6 * NRING, r = G::nth(c, q < 0 ? 0 : q);
        const bool conv = q < 0, dx = q >= 0 && q < G::share(3) && r < 3;
        if (conv || dx) {
            C *z = conv ? B + grp * RC : X + q * RC;
            const C *__restrict__ src =
                spec + (size_t)(conv ? c * CHN + rr * 8 + ring_dir(grp - 6 * rr) : SLOT_X + r) * slot;
            row_pre<H, 1>(z, TB.wp, j, src, src, [](int, C a, C) { return a; }, ready);
            __syncwarp(lanes_of_row<P>());
            row_fft<H, +1>(z, TB.tw, j);
            if constexpr (CS > 1) {
                fence_proxy_async();
                __syncwarp(lanes_of_row<P>());
            }
        }
        ready();   // (no copy is in flight when the block ends)
        row_gone<CS>();
        // the d_x rows' slices into the first three rows of co, each to the
        // block that replaces them by coefficients
        if (CS > 1 && dx && j < CS)
            push_bulk(co + r * NX + j * NXS, reinterpret_cast<const real *>(X + q * RC) + j * NXS, NXS * sizeof(real), &xbar, j);
    }
    if constexpr (CS == 1) __syncthreads();
    else table_wait<true>(&xbar, A.err);
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        real dx[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
            dx[r] = CS == 1 ? reinterpret_cast<const real *>(X + G::local(r) * RC)[x] : co[r * NX + x];
        const real rho = row(SLOT_F)[x], ux = row(SLOT_F + 1)[x], uy = row(SLOT_F + 2)[x], T = row(SLOT_F + 3)[x];
        const real rT = rho * T, irT = real(1) / rT, iT = real(1) / T;
        const real Bx = (row(SLOT_A + 1)[x] + row(SLOT_L2)[x] + dx[1]) * irT;        // Eq. 21
        const real By = (row(SLOT_A + 2)[x] + row(SLOT_L2 + 1)[x] + dx[2]) * irT;
        const real CC = (row(SLOT_A)[x] + row(SLOT_L2 + 2)[x] + dx[0]) * (real(0.5) * irT * iT);   // C + C_q, Eqs. 22-23
        const real At = real(-2) * CC * T;                                          // Eq. 20
        const real u2 = ux * ux + uy * uy;
        // I = -(A + B.(v-u) + CC |v-u|^2) f^eq = -(e0 + e1.v + CC |v|^2) f^eq
        const real e[NCOEF] = {At - (Bx * ux + By * uy) + CC * u2, Bx - real(2) * CC * ux, By - real(2) * CC * uy, CC, iT};
#pragma unroll
        for (int i = 0; i < NCOEF; ++i) co[i * NX + x] = e[i];
    }
    if constexpr (CS > 1) fence_proxy_async();
    __syncthreads();
    if (CS > 1 && tid < (CS - 1) * NCOEF) {
        const int i = tid / (CS - 1), b = tid - i * (CS - 1);
        real *q = co + i * NX + c * NXS;
        push_bulk(q, q, NXS * sizeof(real), &cbar, b < c ? b : b + 1);
    }
    // the rest velocity (no convection) at this block's slice
    for (int x = c * NXS + tid; x < (c + 1) * NXS; x += NT) {
        const real rho = row(SLOT_F)[x], ux = row(SLOT_F + 1)[x], uy = row(SLOT_F + 2)[x], T = row(SLOT_F + 3)[x];
        const real fc = A.fcur[fo + x];
        real F0 = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) F0 += wk(A, k, T);
        F0 = real(1) - real(8) * F0;
        const real qq = real(0.5) * (ux * ux + uy * uy) * co[4 * NX + x], om = real(1) - qq;
        const real fe = rho * F0 * (om + real(0.5) * qq * qq);
        A.fout[fo + x] =
            rk_combine(with_base, beta, dt, fc, with_base ? A.fbase[fo + x] : real(0), -(fc - fe) * itau - co[x] * fe);
    }
    if constexpr (CS > 1) table_wait<true>(&cbar, A.err);
    row_leave<CS>();   // (nothing more comes; its own slices may still be on their way)
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
        real rho[V], ux[V], uy[V], T[V], e0[V], ex[V], ey[V], CC[V], iT[V];
        ldv<real, V>(rho, row(SLOT_F) + x);
        ldv<real, V>(ux, row(SLOT_F + 1) + x);
        ldv<real, V>(uy, row(SLOT_F + 2) + x);
        ldv<real, V>(T, row(SLOT_F + 3) + x);
        ldv<real, V>(e0, co + x);
        ldv<real, V>(ex, co + NX + x);
        ldv<real, V>(ey, co + 2 * NX + x);
        ldv<real, V>(CC, co + 3 * NX + x);
        ldv<real, V>(iT, co + 4 * NX + x);
        const real hh = real(0.70710678118654752440);
        real p0[V], p1[V], p2[V], p3[V], p4[V], h0[V], dp[V], dm[V], ep[V], em[V];
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
            h0[q] = e0[q] + CC[q] * sk2;
            ux[q] *= sk;
            uy[q] *= sk;
            ex[q] *= sk;
            ey[q] *= sk;
            dp[q] = hh * (ux[q] + uy[q]);
            dm[q] = hh * (uy[q] - ux[q]);
            ep[q] = hh * (ex[q] + ey[q]);
            em[q] = hh * (ey[q] - ex[q]);
        }
        const real *cr = reinterpret_cast<const real *>(B + rr * 6 * RC) + x;
        // directions r and r + 4 together: f^eq = even +- odd in v.u
#pragma unroll
        for (int r0 = 0; r0 < 4; r0 += RP) {
            real fc[2 * RP][V], fb[2 * RP][V], cv[2 * RP][V];
            // (a direction's loads come before its stores: fout may be fcur or
            // fbase, at the same site)
#pragma unroll
            for (int q = 0; q < 2 * RP; ++q) {
                const int r = r0 + (q >> 1) + 4 * (q & 1);
                ldv<real, V>(fc[q], pc + (size_t)r * N);
                if (with_base) ldv_once<real, V>(fb[q], pb + (size_t)r * N);
                if ((r & 3) == 2) ldv<real, V>(cv[q], row(v0 + r) + x);   // v_x = 0: real from the column pass
                else ldv<real, V>(cv[q], cr + (size_t)ring_pos(r) * 2 * RC);
            }
#pragma unroll
            for (int h = 0; h < RP; ++h) {
                const int r = r0 + h;
                real fn[2][V];
#pragma unroll
                for (int q = 0; q < V; ++q) {
                    const real vu = ring_dot<real>(r, ux[q], uy[q], dp[q], dm[q]), w2 = vu * vu;
                    const real ev = p0[q] + w2 * (p2[q] + w2 * p4[q]), od = vu * (p1[q] + w2 * p3[q]);   // Eq. 3
                    const real ed = ring_dot<real>(r, ex[q], ey[q], ep[q], em[q]);
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        const real fe = s ? ev - od : ev + od;
                        // -(f - f^eq) / tau - g f^eq - convection, g = -I / f^eq (Eqs. 10, 11);
                        // the difference before its product with 1 / tau: as (1 / tau - g)
                        // f^eq - f / tau it is an operation less and rounds f dt / tau twice
                        const real g = s ? h0[q] - ed : h0[q] + ed;
                        const real f = fc[2 * h + s][q];
                        const real rhs = -(f - fe) * itau - cv[2 * h + s][q] - g * fe;
                        fn[s][q] = rk_combine(with_base, beta, dt, f, fb[2 * h + s][q], rhs);
                    }
                }
                stv_once<real, V>(po + (size_t)r * N, fn[0]);
                stv_once<real, V>(po + (size_t)(r + 4) * N, fn[1]);
            }
        }
    }
    row_gone<CS>();
}

template <typename real, int H> size_t k5_row_smem() {
    using G = Row<real, H>;
    return (size_t)(6 * G::NRING + G::share(3)) * G::RC * 2 * sizeof(real) + (size_t)NCOEF * G::NX * sizeof(real) +
           RowTable<real>::bytes(H) - RowTable<real>::tw(H);
}

// ---------------------------------------------------------------------------
// Single rows: one row per row group, NG rows per block, no cluster.
// ---------------------------------------------------------------------------

// Half-length transform Z of a real row -> the packed half-length spectrum of
// its d_x (i k_x X / nx), in place: row_post, the product and row_pre pair by
// pair.
template <int H, typename C>
__device__ __forceinline__ void row_dx(C *z, const C *wh, const C *wp, const decltype(C::x) *kx, int j) {
    using R = decltype(z[0].x);
    constexpr int P = Row<R, H>::P;
    static_assert(H % (2 * P) == 0, "row configuration");
    const R sx = R(1.0 / (2 * H));
#pragma unroll
    for (int k0 = 0; k0 < H / 2; k0 += P) {
        const int k = k0 + j;
        if (k == 0) {   // bins 0 and H / 2: Y = i m conj z, Z = 2 conj Y
            z[0] = C{0, 0};
            const C zh = z[H / 2];
            const R m = R(2) * (kx[H / 2] * sx);
            z[H / 2] = C{m * zh.y, -m * zh.x};
        } else {
            const C p = z[k], q = z[H - k];
            const C s = cadd(p, cconj(q)), d = csub(p, cconj(q));
            const C w = cmul(wh[k], cmul_mi(d));
            const R m = kx[k] * sx, mh = kx[H - k] * sx;
            // X[k] = s/2 + w, X[H-k] = conj(s/2 - w); Y = i m X
            const C yk = C{-m * (R(0.5) * s.y + w.y), m * (R(0.5) * s.x + w.x)};
            const C yc = C{mh * (R(0.5) * s.y - w.y), -mh * (R(0.5) * s.x - w.x)};   // conj Y[H-k]
            const C a = cadd(yk, yc), e = csub(yk, yc);
            const C t = cmul_i(cmul(e, cconj(wp[k])));
            z[k] = cadd(a, t);
            z[H - k] = cconj(csub(a, t));
        }
    }
}

// tables [0, bytes) behind the NG rows of a single-row kernel
template <typename real, int H>
__device__ __forceinline__ bool single_tables(unsigned char *tb, const typename Row<real, H>::C *tab, uint64_t *bar, int *err) {
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_init_fence();
        mbar_expect_tx(bar, RowTable<real>::bytes(H));
        table_issue(tb, tab, 0, RowTable<real>::bytes(H), bar);
    }
    __syncthreads();
    if (block_wait(bar, 0, err)) return true;
    mbar_wait_bounded(bar, 0);
    return false;
}

// D_x of caller fields g (fp64 rows) into out[2 field]: a derivative along x
// needs the row's own transforms and nothing else.
template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) dx_row(const __grid_constant__ GradArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int P = G::P;
    extern __shared__ __align__(128) unsigned char row_smem[];
    __shared__ __align__(8) uint64_t bar;
    C *B = reinterpret_cast<C *>(row_smem);
    unsigned char *tb = reinterpret_cast<unsigned char *>(B + G::NG * G::RC);
    const Tab<real, H> T(tb, 0);
    const int tid = threadIdx.x, j = tid & (P - 1), grp = tid / P, r = (int)blockIdx.x * G::NG + grp;
    const bool mine = r < A.nrows;
    C *z = B + grp * G::RC;
    if (mine) {
        const double2 *__restrict__ in = A.g + (size_t)r * H;
        double2 x[G::E];
#pragma unroll
        for (int t = 0; t < G::E; ++t) x[t] = in[j + P * t];
#pragma unroll
        for (int t = 0; t < G::E; ++t) z[j + P * t] = C{(real)x[t].x, (real)x[t].y};
    }
    if (!single_tables<real, H>(tb, A.rtab, &bar, A.err)) return;
    if (!mine) return;
    row_fft<H, -1>(z, T.tw, j);
    row_dx<H>(z, T.wh, T.wp, T.kx, j);
    __syncwarp(lanes_of_row<P>());
    row_fft<H, +1>(z, T.tw, j);
    const int field = r / A.ny, y = r - field * A.ny;
    double2 *out = A.out + ((size_t)2 * field * A.ny + y) * H;
#pragma unroll
    for (int t = 0; t < G::E; ++t) {
        const C w = z[j + P * t];
        out[j + P * t] = make_double2((double)w.x, (double)w.y);
    }
}

// Sum over the block's rows of (D_x rho)^2 by Parseval's relation: over the
// two-sided spectrum sum_x d^2 = (1 / nx) sum_k |i k_x X_k|^2.
template <typename real, int H>
__global__ void __launch_bounds__(Row<real, H>::NT, row_minb<real, H>()) energy_row(const __grid_constant__ EnergyArgs<real> A) {
    using G = Row<real, H>;
    using C = typename G::C;
    constexpr int P = G::P;
    extern __shared__ __align__(128) unsigned char row_smem[];
    __shared__ __align__(8) uint64_t bar;
    C *B = reinterpret_cast<C *>(row_smem);
    unsigned char *tb = reinterpret_cast<unsigned char *>(B + G::NG * G::RC);
    const Tab<real, H> T(tb, 0);
    const int tid = threadIdx.x, j = tid & (P - 1), grp = tid / P, y = (int)blockIdx.x * G::NG + grp;
    const bool mine = y < A.ny;
    C *z = B + grp * G::RC;
    grid_dep_wait();
    if (mine) {
        const C *__restrict__ in = A.rho + (size_t)y * H;
#pragma unroll
        for (int t = 0; t < G::E; ++t) z[j + P * t] = in[j + P * t];
    }
    if (!single_tables<real, H>(tb, A.rtab, &bar, A.err)) return;
    double e = 0;
    if (mine) {
        row_fft<H, -1>(z, T.tw, j);
        row_post<H>(z, T.wh, j, [&](int k, C X) {
            if (k > 0) {
                const real m = T.kx[k];
                e += 2.0 * (double)(m * m * (X.x * X.x + X.y * X.y));
            }
        });
    }
    block_sum_store<G::NT>(e * (1.0 / (2 * H)), A.partial_x + blockIdx.x);
}

template <typename real, int H> RowSet row_set() {
    using G = Row<real, H>;
    RowSet s;
    s.k1 = (const void *)&k1_row<real, H>;
    s.k3 = (const void *)&k3_row<real, H>;
    s.k5 = (const void *)&k5_row<real, H>;
    s.dx = (const void *)&dx_row<real, H>;
    s.energy = (const void *)&energy_row<real, H>;
    s.ng = G::NG;
    s.smem_rows = (size_t)G::NG * G::RC * 2 * sizeof(real) + RowTable<real>::bytes(H);
    s.nt = G::NT;
    s.nt3 = row_nt3((int)sizeof(real), H);
    s.cs = G::CS;
    s.smem1 = k1_row_smem<real, H>();
    s.smem3 = k3_row_smem<real, H>();
    s.smem5 = k5_row_smem<real, H>();
    return s;
}

}  // namespace rk

}  // namespace fftlb

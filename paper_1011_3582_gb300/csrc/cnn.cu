// Learned warm start (include/fftlb_warmstart.h): a 4-layer periodic 3x3
// convolutional network trained on FFT-LB snapshots (arXiv:1011.3582,
// Sec. 4 phase separation) and applied to a handle's state.
//
// Every convolution is an implicit GEMM on the tensor cores: bfloat16
// operands staged in shared memory, mma.sync m16n8k16 with fp32
// accumulators.  Activations are NHWC bfloat16 (channels padded to 16 or
// 32), so one pixel's channels are contiguous 16-byte chunks.  Tiles are 64
// pixels x 4 rows with a one-pixel halo, staged by cp.async two deep (the next
// tile lands while this one is multiplied); fragments come by ldmatrix, from
// pixel rows padded by 8 channels (conflict-free):
//   k_conv<CIN, COUT, FWD_RELU | FWD_LAST | BWD>
//       out[p][n] = sum_tap sum_k w[tap][n][k] in[p + d(tap)][k]
//       FWD: + bias, ReLU (layers 1-3, bfloat16 out) or fp32 planar out
//       (layer 4).  BWD: the input gradient, using the weights transposed
//       and flipped (d -> -d), times the ReLU mask of the stored activation.
//   k_wgrad<CIN, GC>: dW[co][tap][ci] = sum_p G[p][co] A[p + d(tap)][ci] and
//       db[co] = sum_p G[p][co] (M = co, N = ci, K = pixels), one partial sum
//       per block; k_update adds the blocks' partials in order (no atomics: a
//       gradient is reproducible) and applies Adam.
// Measured at 512^2 (a training step 800 -> 299 us): k_conv<32, 32> 36 ->
// 19 us (a warp held 16 pixels and loaded every weight fragment for them
// alone, three 4-byte shared loads a product), k_wgrad<32, 32> 156 -> 28 us
// (fragments gathered from 2-byte loads, one 4-warp block per SM), the bias
// gradients' own pass over G (17 us a layer) gone.
// The parameter gradient, loss and Adam state are fp32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/fftlb_warmstart.h"
#include "engine.h"

namespace {

using bf16 = __nv_bfloat16;

constexpr int NL = 4;
// channels per layer l = 0..3 (functions so that host and device code share them)
__host__ __device__ constexpr int CIN_R(int l) { return l == 0 ? 3 : 32; }     // real input
__host__ __device__ constexpr int COUT_R(int l) { return l == 3 ? 2 : 32; }    // real output
__host__ __device__ constexpr int CINP(int l) { return l == 0 ? 16 : 32; }     // padded input (forward)
__host__ __device__ constexpr int COUTP(int l) { return l == 3 ? 8 : 32; }     // padded output (forward)
__host__ __device__ constexpr int GCH(int l) { return l == 3 ? 16 : 32; }      // stored gradient G_l
constexpr int TX = 64;                        // pixels per tile row
constexpr int RT = 4;                         // rows per tile
constexpr int NTC = 256;                      // k_conv: 8 warps, (row, half row) each: 32 pixels
constexpr int NTW = 384;                      // k_wgrad: 12 warps, (tap row, tile row) each

enum { FWD_RELU = 0, FWD_LAST = 1, BWD = 2 };

__host__ __device__ constexpr int w_size(int l) { return COUT_R(l) * 9 * CIN_R(l); }
__host__ __device__ constexpr int w_off(int l) { return l == 0 ? 0 : w_off(l - 1) + w_size(l - 1) + COUT_R(l - 1); }
__host__ __device__ constexpr int b_off(int l) { return w_off(l) + w_size(l); }
static_assert(b_off(NL - 1) + COUT_R(NL - 1) == FFTLB_CNN_NPARAMS, "parameter layout");

__device__ __forceinline__ void mma_bf16(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ uint32_t sm32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(sm32(p)) : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], const bf16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(sm32(p)) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(sm32(p)) : "memory");
}
__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sm32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// row i of a periodic axis of n, -1 <= i; rows past n (only those below a
// ragged last tile's halo) give some valid row
__device__ __forceinline__ int wrap_row(int i, int n) { return i < 0 ? i + n : i < n ? i : i - n < n ? i - n : 0; }

// stage rows y-1 .. y+RT, pixels x0-1 .. x0+TX of an NHWC bfloat16 tensor with C
// channels into s[RT + 2][TX + 2][C + 8] (periodic)
template <int C, int NTHR>
__device__ __forceinline__ void stage_halo(bf16 *s, const bf16 *in, int y, int x0, int H, int W) {
    constexpr int CH = C / 8, PX = TX + 2;
    for (int i = threadIdx.x; i < (RT + 2) * PX * CH; i += NTHR) {
        const int ch = i % CH, px = (i / CH) % PX, r = i / (CH * PX);
        const int yy = wrap_row(y + r - 1, H), xr = x0 + px - 1, xx = xr < 0 ? xr + W : xr >= W ? xr - W : xr;
        cp16(s + (size_t)(r * PX + px) * (C + 8) + ch * 8, in + ((size_t)yy * W + xx) * C + ch * 8);
    }
}

template <int CIN, int COUT> constexpr size_t conv_smem() {
    return sizeof(bf16) * (CIN + 8) * (9 * COUT + 2 * (RT + 2) * (TX + 2));
}

template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(NTC, 2) k_conv(const bf16 *__restrict__ in, const bf16 *__restrict__ w,
                                                 const float *__restrict__ bias, void *out,
                                                 const bf16 *__restrict__ mask, int H, int W) {
    constexpr int SC = CIN + 8, PX = TX + 2, BUF = (RT + 2) * PX * SC;
    constexpr int NT = COUT / 8, MT = 2;
    extern __shared__ __align__(16) unsigned char cnn_smem[];
    bf16 *w_s = reinterpret_cast<bf16 *>(cnn_smem);   // [9][COUT][SC]
    bf16 *in_s = w_s + 9 * COUT * SC;                 // [2][RT + 2][PX][SC]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int row = warp >> 1, px0 = (warp & 1) * 32;
    const int tpr = W / TX, ntiles = (H + RT - 1) / RT * tpr;
    const size_t P = (size_t)H * W;
    // this lane's ldmatrix rows: A (pixels x channels), B (outputs x channels)
    const int la = (lane & 7) + ((lane >> 3) & 1) * 8, ka = (lane >> 4) * 8;
    const int lb = (lane & 7) + (lane >> 4) * 8, kb = ((lane >> 3) & 1) * 8;
    for (int i = threadIdx.x; i < 9 * COUT * (CIN / 8); i += NTC) {
        const int r = i / (CIN / 8), ch = i % (CIN / 8);
        cp16(w_s + (size_t)r * SC + ch * 8, w + (size_t)r * CIN + ch * 8);
    }
    int tile = blockIdx.x;
    if (tile < ntiles) stage_halo<CIN, NTC>(in_s, in, tile / tpr * RT, tile % tpr * TX, H, W);
    cp_commit();
    for (int b = 0; tile < ntiles; tile += gridDim.x, b ^= 1) {
        const int next = tile + gridDim.x;
        if (next < ntiles) stage_halo<CIN, NTC>(in_s + (b ^ 1) * BUF, in, next / tpr * RT, next % tpr * TX, H, W);
        cp_commit();
        cp_wait<1>();
        __syncthreads();
        const int y = tile / tpr * RT + row, x0 = tile % tpr * TX + px0;
        const bf16 *s = in_s + b * BUF;
        if (y < H) {   // (uniform over the warp)
            float acc[MT][NT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) acc[m][nt][0] = acc[m][nt][1] = acc[m][nt][2] = acc[m][nt][3] = 0.f;
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const bf16 *a0 = s + (size_t)((row + tap / 3) * PX + px0 + tap % 3 + la) * SC + ka;
#pragma unroll
                for (int kc = 0; kc < CIN / 16; ++kc) {
                    uint32_t a[MT][4];
#pragma unroll
                    for (int m = 0; m < MT; ++m) ldsm4(a[m], a0 + (size_t)m * 16 * SC + kc * 16);
                    uint32_t bb[NT][2];
                    const bf16 *wt = w_s + (size_t)tap * COUT * SC + kc * 16;
                    if constexpr (NT == 1) {
                        ldsm2(bb[0], wt + (size_t)(lane & 7) * SC + kb);
                    } else {
#pragma unroll
                        for (int n2 = 0; n2 < NT / 2; ++n2) {
                            uint32_t q[4];
                            ldsm4(q, wt + (size_t)(n2 * 16 + lb) * SC + kb);
                            bb[2 * n2][0] = q[0];
                            bb[2 * n2][1] = q[1];
                            bb[2 * n2 + 1][0] = q[2];
                            bb[2 * n2 + 1][1] = q[3];
                        }
                    }
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt)
                            mma_bf16(acc[m][nt], a[m][0], a[m][1], a[m][2], a[m][3], bb[nt][0], bb[nt][1]);
                }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const size_t pa = (size_t)y * W + x0 + m * 16 + g, pb = pa + 8;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const int co = nt * 8 + 2 * t;
                    const float *c4 = acc[m][nt];
                    if (MODE == FWD_RELU) {
                        bf16 *o = reinterpret_cast<bf16 *>(out);
                        const float b0 = bias[co], b1 = bias[co + 1];
                        *reinterpret_cast<__nv_bfloat162 *>(o + pa * COUT + co) =
                            __floats2bfloat162_rn(fmaxf(c4[0] + b0, 0.f), fmaxf(c4[1] + b1, 0.f));
                        *reinterpret_cast<__nv_bfloat162 *>(o + pb * COUT + co) =
                            __floats2bfloat162_rn(fmaxf(c4[2] + b0, 0.f), fmaxf(c4[3] + b1, 0.f));
                    } else if (MODE == FWD_LAST) {
                        float *o = reinterpret_cast<float *>(out);
                        if (co < 2) {   // two real output channels, planar
                            o[(size_t)co * P + pa] = c4[0] + bias[co];
                            o[(size_t)(co + 1) * P + pa] = c4[1] + bias[co + 1];
                            o[(size_t)co * P + pb] = c4[2] + bias[co];
                            o[(size_t)(co + 1) * P + pb] = c4[3] + bias[co + 1];
                        }
                    } else {
                        bf16 *o = reinterpret_cast<bf16 *>(out);
                        const __nv_bfloat162 ma = *reinterpret_cast<const __nv_bfloat162 *>(mask + pa * COUT + co);
                        const __nv_bfloat162 mb = *reinterpret_cast<const __nv_bfloat162 *>(mask + pb * COUT + co);
                        *reinterpret_cast<__nv_bfloat162 *>(o + pa * COUT + co) = __floats2bfloat162_rn(
                            __low2float(ma) > 0.f ? c4[0] : 0.f, __high2float(ma) > 0.f ? c4[1] : 0.f);
                        *reinterpret_cast<__nv_bfloat162 *>(o + pb * COUT + co) = __floats2bfloat162_rn(
                            __low2float(mb) > 0.f ? c4[2] : 0.f, __high2float(mb) > 0.f ? c4[3] : 0.f);
                    }
                }
            }
        }
        __syncthreads();   // this buffer is refilled next
    }
    cp_wait<0>();
}

// One layer's partial sums of a block in the workspace: dW as [tap][co][ci]
// (GC x CIN, padded channels included), then db [GC]
template <int CIN, int GC> constexpr int wg_size() { return 9 * GC * CIN + GC; }
template <int CIN, int GC> constexpr size_t wgrad_smem() {
    return 2 * sizeof(bf16) * ((RT + 2) * (TX + 2) * (CIN + 8) + RT * TX * (GC + 8));
}

// ws[block] = this block's sum over its tiles of G[p][co] A[p + d(tap)][ci] and
// of G[p][co]; warp (ky, r) takes the taps (ky, 0..2) at row r of each tile.
template <int CIN, int GC>
__global__ void __launch_bounds__(NTW, 1) k_wgrad(const bf16 *__restrict__ G, const bf16 *__restrict__ A,
                                                  float *__restrict__ ws, int H, int W) {
    constexpr int SA = CIN + 8, SG = GC + 8, PX = TX + 2;
    constexpr int ABUF = (RT + 2) * PX * SA, GBUF = RT * TX * SG;
    constexpr int MT = GC / 16, NT = CIN / 8;
    extern __shared__ __align__(16) unsigned char cnn_smem[];
    bf16 *a_s = reinterpret_cast<bf16 *>(cnn_smem);   // [2][RT + 2][PX][SA]
    bf16 *g_s = a_s + 2 * ABUF;                       // [2][RT][TX][SG]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int ky = warp % 3, row = warp / 3;
    const int tpr = W / TX, ntiles = (H + RT - 1) / RT * tpr;
    // this lane's ldmatrix rows (pixels) and channel offsets: G as the A operand
    // (co x pixel), A as the B operand (pixel x ci), both transposed on the way
    const int pg = (lane & 7) + (lane >> 4) * 8, cg_ = ((lane >> 3) & 1) * 8;
    const int pa = (lane & 7) + ((lane >> 3) & 1) * 8, ca = (lane >> 4) * 8;
    auto stage = [&](int tile, int b) {
        const int y = tile / tpr * RT, x0 = tile % tpr * TX;
        stage_halo<CIN, NTW>(a_s + b * ABUF, A, y, x0, H, W);
        constexpr int CH = GC / 8;
        for (int i = threadIdx.x; i < RT * TX * CH; i += NTW) {
            const int ch = i % CH, px = (i / CH) % TX, r = i / (CH * TX);
            if (y + r < H)
                cp16(g_s + b * GBUF + (size_t)(r * TX + px) * SG + ch * 8, G + ((size_t)(y + r) * W + x0 + px) * GC + ch * 8);
        }
    };
    float acc[3][MT][NT][4], accb[MT][4];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NT; ++n) acc[j][m][n][0] = acc[j][m][n][1] = acc[j][m][n][2] = acc[j][m][n][3] = 0.f;
#pragma unroll
    for (int m = 0; m < MT; ++m) accb[m][0] = accb[m][1] = accb[m][2] = accb[m][3] = 0.f;
    int tile = blockIdx.x;
    if (tile < ntiles) stage(tile, 0);
    cp_commit();
    for (int b = 0; tile < ntiles; tile += gridDim.x, b ^= 1) {
        const int next = tile + gridDim.x;
        if (next < ntiles) stage(next, b ^ 1);
        cp_commit();
        cp_wait<1>();
        __syncthreads();
        if (tile / tpr * RT + row < H) {   // (uniform over the warp)
            const bf16 *gs = g_s + b * GBUF + (size_t)(row * TX + pg) * SG + cg_;
            const bf16 *as = a_s + b * ABUF + (size_t)((row + ky) * PX + pa) * SA + ca;
#pragma unroll
            for (int ks = 0; ks < TX / 16; ++ks) {
                uint32_t a[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m) ldsm4t(a[m], gs + (size_t)ks * 16 * SG + m * 16);
                if (ky == 0) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(accb[m], a[m][0], a[m][1], a[m][2], a[m][3], 0x3f803f80u, 0x3f803f80u);
                }
#pragma unroll
                for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                    for (int n2 = 0; n2 < NT / 2; ++n2) {
                        uint32_t q[4];
                        ldsm4t(q, as + (size_t)(ks * 16 + kx) * SA + n2 * 16);
#pragma unroll
                        for (int m = 0; m < MT; ++m) {
                            mma_bf16(acc[kx][m][2 * n2], a[m][0], a[m][1], a[m][2], a[m][3], q[0], q[1]);
                            mma_bf16(acc[kx][m][2 * n2 + 1], a[m][0], a[m][1], a[m][2], a[m][3], q[2], q[3]);
                        }
                    }
            }
        }
        __syncthreads();   // this buffer is refilled next
    }
    cp_wait<0>();
    __syncthreads();
    // the tile rows' sums one after another into shared memory, then out
    float *red = reinterpret_cast<float *>(cnn_smem);
    static_assert(sizeof(float) * wg_size<CIN, GC>() <= wgrad_smem<CIN, GC>(), "reduction buffer");
    for (int r = 0; r < RT; ++r) {
        if (row == r) {
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int co = m * 16 + g + (e >= 2 ? 8 : 0), ci = n * 8 + 2 * t + (e & 1);
                            float *p = red + ((size_t)(ky * 3 + kx) * GC + co) * CIN + ci;
                            *p = r == 0 ? acc[kx][m][n][e] : *p + acc[kx][m][n][e];
                        }
            if (ky == 0 && t == 0)
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int e = 0; e < 4; e += 2) {
                        float *p = red + (size_t)9 * GC * CIN + m * 16 + g + (e ? 8 : 0);
                        *p = r == 0 ? accb[m][e] : *p + accb[m][e];
                    }
        }
        __syncthreads();
    }
    float *o = ws + (size_t)blockIdx.x * wg_size<CIN, GC>();
    for (int i = threadIdx.x; i < wg_size<CIN, GC>(); i += NTW) o[i] = red[i];
}

// A0[p][c] = bf16(X[c][p]) for c < 3, channels 3..15 zero
__global__ void k_prep(const float *__restrict__ X, bf16 *__restrict__ A0, size_t P) {
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P; p += (size_t)gridDim.x * blockDim.x) {
        const bf16 z = __float2bfloat16_rn(0.f);
        uint4 lo;
        lo.x = pack2(__float2bfloat16_rn(X[p]), __float2bfloat16_rn(X[P + p]));
        lo.y = pack2(__float2bfloat16_rn(X[2 * P + p]), z);
        lo.z = lo.w = 0u;
        uint4 *d = reinterpret_cast<uint4 *>(A0 + p * 16);
        d[0] = lo;
        d[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// residual R = Y - (Xt - X[0:2]); part[block] = sum R^2 / n; G4[p][c] = bf16(2 R /
// n), channels 2..15 zero (whole 32-byte sectors)
__global__ void __launch_bounds__(256) k_loss(const float *__restrict__ Y, const float *__restrict__ X,
                                              const float *__restrict__ Xt, bf16 *__restrict__ G4, double *part, size_t P) {
    __shared__ double red[8];
    const double inv_n = 1.0 / (2.0 * (double)P);
    double s = 0.0;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P; p += (size_t)gridDim.x * blockDim.x) {
        const float r0 = Y[p] - (Xt[p] - X[p]);
        const float r1 = Y[P + p] - (Xt[P + p] - X[P + p]);
        s += (double)r0 * r0 + (double)r1 * r1;
        uint4 *d = reinterpret_cast<uint4 *>(G4 + p * 16);
        d[0] = make_uint4(pack2(__float2bfloat16_rn((float)(2.0 * r0 * inv_n)), __float2bfloat16_rn((float)(2.0 * r1 * inv_n))),
                          0u, 0u, 0u);
        d[1] = make_uint4(0u, 0u, 0u, 0u);
    }
    for (int w = 16; w > 0; w >>= 1) s += __shfl_down_sync(0xffffffffu, s, w);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += red[w];
        part[blockIdx.x] = s * inv_n;
    }
}

struct WeightPtrs {
    bf16 *wf[NL];   // [9][COUTP][CINP]
    bf16 *wb[NL];   // layers 2..4: [9][CIN_R = 32][GCH] (flipped taps, transposed)
    float *bias[NL];
};

// bfloat16 weight tiles for the forward and backward kernels from the fp32
// parameter vector (one thread per tile entry)
__global__ void k_weights(const float *__restrict__ prm, WeightPtrs wp) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int r = i;
    for (int l = 0; l < NL; ++l) {
        const int nf = 9 * COUTP(l) * CINP(l);
        if (r < nf) {
            const int ci = r % CINP(l), co = (r / CINP(l)) % COUTP(l), tap = r / (CINP(l) * COUTP(l));
            const float v = (co < COUT_R(l) && ci < CIN_R(l)) ? prm[w_off(l) + (co * 9 + tap) * CIN_R(l) + ci] : 0.f;
            wp.wf[l][r] = __float2bfloat16_rn(v);
            return;
        }
        r -= nf;
        if (l > 0) {
            const int nb = 9 * CIN_R(l) * GCH(l);
            if (r < nb) {
                const int co = r % GCH(l), ci = (r / GCH(l)) % CIN_R(l), tp = r / (GCH(l) * CIN_R(l));
                const float v = co < COUT_R(l) ? prm[w_off(l) + (co * 9 + (8 - tp)) * CIN_R(l) + ci] : 0.f;
                wp.wb[l][r] = __float2bfloat16_rn(v);
                return;
            }
            r -= nb;
        }
        if (r < COUTP(l)) {
            wp.bias[l][r] = r < COUT_R(l) ? prm[b_off(l) + r] : 0.f;
            return;
        }
        r -= COUTP(l);
    }
}

int weight_entries() {
    int n = 0;
    for (int l = 0; l < NL; ++l) n += 9 * COUTP(l) * CINP(l) + (l > 0 ? 9 * CIN_R(l) * GCH(l) : 0) + COUTP(l);
    return n;
}

// where each layer's partials sit in the workspace (nblk blocks of wgn[l] floats
// from off[l]), and the loss partials
struct GradParts {
    const float *ws;
    size_t off[NL];
    int wgn[NL], nblk;
    const double *loss_part;
    int nloss;
};
// row length (channels of A) and rows (channels of G) of layer l's partials
__host__ __device__ constexpr int WGC(int l) { return CINP(l); }
__host__ __device__ constexpr int WGG(int l) { return GCH(l); }

// Parameter gradients from the blocks' partials, summed in block order by the 8
// threads of a parameter (interleaved, then in order), the loss, and with adam
// one Adam step and the bfloat16 weight tiles of the new parameters.  32
// parameters per block.
__global__ void __launch_bounds__(256) k_update(GradParts gp, float *__restrict__ grad, double *loss, int adam,
                                                float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                                                float lr, float bc1, float bc2, WeightPtrs wp) {
    __shared__ float red[8][33];
    __shared__ double lred[8];
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    if (blockIdx.x == 0) {
        double s = 0;
        for (int b = threadIdx.x; b < gp.nloss; b += 256) s += gp.loss_part[b];
        for (int q = 16; q > 0; q >>= 1) s += __shfl_down_sync(0xffffffffu, s, q);
        if (lane == 0) lred[seg] = s;
    }
    int l = 0, r = i;
    while (l < NL - 1 && r >= w_size(l) + COUT_R(l)) r -= w_size(l) + COUT_R(l), ++l;
    const bool ok = i < FFTLB_CNN_NPARAMS, isb = r >= w_size(l);
    int co = 0, tap = 0, ci = 0, at = 0;
    if (ok) {
        if (isb) {
            co = r - w_size(l);
            at = 9 * WGG(l) * WGC(l) + co;
        } else {
            ci = r % CIN_R(l);
            tap = (r / CIN_R(l)) % 9;
            co = r / (9 * CIN_R(l));
            at = (tap * WGG(l) + co) * WGC(l) + ci;
        }
    }
    float s = 0.f;
    if (ok) {
        const float *p = gp.ws + gp.off[l] + at;
#pragma unroll 4
        for (int b = seg; b < gp.nblk; b += 8) s += p[(size_t)b * gp.wgn[l]];
    }
    red[seg][lane] = s;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0 && loss) {
        double t = lred[0];
        for (int q = 1; q < 8; ++q) t += lred[q];
        *loss = t;
    }
    if (seg || !ok) return;
    float gi = red[0][lane];
    for (int q = 1; q < 8; ++q) gi += red[q][lane];
    grad[i] = gi;
    if (!adam) return;
    const float mi = 0.9f * m[i] + 0.1f * gi, vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wn = w[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + 1e-8f);
    w[i] = wn;
    if (isb) {
        wp.bias[l][co] = wn;
    } else {   // (the tiles' padding stays zero)
        const bf16 h = __float2bfloat16_rn(wn);
        wp.wf[l][(tap * COUTP(l) + co) * CINP(l) + ci] = h;
        if (l > 0) wp.wb[l][((8 - tap) * CIN_R(l) + ci) * GCH(l) + co] = h;
    }
}

__global__ void k_encode(const double *__restrict__ rho, const double *__restrict__ T, float *__restrict__ X,
                         size_t P, double rho_c, double T_c, double s_rho, double s_T, double T_run) {
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P; p += (size_t)gridDim.x * blockDim.x) {
        X[p] = (float)(s_rho * (rho[p] / rho_c - 1.0));
        X[P + p] = (float)(s_T * (T[p] / T_run - 1.0));
        X[2 * P + p] = (float)(T_run / T_c - 0.75);
    }
}

__global__ void k_decode(const float *__restrict__ X, const float *__restrict__ Y, double *__restrict__ rho,
                         double *__restrict__ u, double *__restrict__ T, size_t P, double rho_c, double s_rho,
                         double s_T, double T_run) {
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P; p += (size_t)gridDim.x * blockDim.x) {
        rho[p] = rho_c * (1.0 + ((double)X[p] + (double)Y[p]) / s_rho);
        T[p] = T_run * (1.0 + ((double)X[P + p] + (double)Y[P + p]) / s_T);
        u[p] = 0.0;
    }
}

}  // namespace

struct fftlb_cnn_s {
    int H = 0, W = 0;
    size_t P = 0;
    cudaStream_t stream = nullptr;
    std::vector<void *> allocs;
    float *prm = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
    float *X = nullptr, *Xt = nullptr, *Y = nullptr;
    float *ws = nullptr;   // wgrad partials of every layer
    double *loss_part = nullptr;
    GradParts gp{};
    bf16 *A[NL] = {nullptr};   // A_0 (16 ch), A_1..A_3 (32 ch)
    bf16 *G[NL] = {nullptr};   // G_1..G_3 (32 ch) in G[0..2], G_4 (16 ch) in G[3]
    double *loss = nullptr, *fields = nullptr;
    WeightPtrs wp{};
    int adam_k = 0;
    int grid_conv = 1, grid_wgrad = 1, grid_loss = 1;
    long launches = 0;
    std::string err;
};

namespace {

fftlb_status fail(fftlb_cnn_t c, fftlb_status code, const std::string &msg) {
    if (c) c->err = msg;
    else fftlb::set_handleless_error(msg);
    return code;
}

#define CCU(c, call)                                                                                   \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess) return fail(c, FFTLB_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

#define CLAUNCH(c)                                                                                     \
    do {                                                                                               \
        cudaError_t e_ = cudaGetLastError();                                                           \
        if (e_ != cudaSuccess) return fail(c, FFTLB_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e_)); \
        ++(c)->launches;                                                                               \
    } while (0)

template <typename T> fftlb_status dalloc(fftlb_cnn_t c, T **p, size_t n) {
    void *q = nullptr;
    if (cudaMalloc(&q, n * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return fail(c, FFTLB_ERR_OOM, "cudaMalloc of " + std::to_string(n * sizeof(T)) + " bytes failed");
    }
    c->allocs.push_back(q);
    *p = reinterpret_cast<T *>(q);
    return FFTLB_OK;
}

void release(fftlb_cnn_t c) {
    for (void *p : c->allocs) cudaFree(p);
    c->allocs.clear();
}

int grid1d(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 4096); }

fftlb_status refresh_weights(fftlb_cnn_t c) {
    const int n = weight_entries();
    k_weights<<<(n + 255) / 256, 256, 0, c->stream>>>(c->prm, c->wp);
    CLAUNCH(c);
    return FFTLB_OK;
}

// the device address of a caller's buffer: itself, or its copy in dst
fftlb_status upload(fftlb_cnn_t c, float *dst, const float *src, size_t n, int on_device, const float **dev) {
    if (!src) return fail(c, FFTLB_ERR_ARG, "NULL buffer");
    *dev = src;
    if (on_device) return FFTLB_OK;
    CCU(c, cudaMemcpyAsync(dst, src, n * sizeof(float), cudaMemcpyHostToDevice, c->stream));
    *dev = dst;
    return FFTLB_OK;
}

template <int CIN, int COUT, int MODE>
fftlb_status conv(fftlb_cnn_t c, const bf16 *in, const bf16 *w, const float *bias, void *out, const bf16 *mask) {
    k_conv<CIN, COUT, MODE><<<c->grid_conv, NTC, conv_smem<CIN, COUT>(), c->stream>>>(in, w, bias, out, mask, c->H, c->W);
    CLAUNCH(c);
    return FFTLB_OK;
}
template <int CIN, int GC> fftlb_status wgrad(fftlb_cnn_t c, int l) {
    k_wgrad<CIN, GC><<<c->grid_wgrad, NTW, wgrad_smem<CIN, GC>(), c->stream>>>(c->G[l], c->A[l], c->ws + c->gp.off[l], c->H, c->W);
    CLAUNCH(c);
    return FFTLB_OK;
}

// forward from X (device) into Y (device)
fftlb_status forward(fftlb_cnn_t c, const float *X, float *Y) {
    k_prep<<<grid1d(c->P), 256, 0, c->stream>>>(X, c->A[0], c->P);
    CLAUNCH(c);
    fftlb_status s;
    if ((s = conv<16, 32, FWD_RELU>(c, c->A[0], c->wp.wf[0], c->wp.bias[0], c->A[1], nullptr)) ||
        (s = conv<32, 32, FWD_RELU>(c, c->A[1], c->wp.wf[1], c->wp.bias[1], c->A[2], nullptr)) ||
        (s = conv<32, 32, FWD_RELU>(c, c->A[2], c->wp.wf[2], c->wp.bias[2], c->A[3], nullptr)) ||
        (s = conv<32, 8, FWD_LAST>(c, c->A[3], c->wp.wf[3], c->wp.bias[3], Y, nullptr)))
        return s;
    return FFTLB_OK;
}

// partial sums of the parameter gradient and the loss for X, Xt (device)
fftlb_status backward(fftlb_cnn_t c, const float *X, const float *Xt) {
    fftlb_status s = forward(c, X, c->Y);
    if (s != FFTLB_OK) return s;
    k_loss<<<c->grid_loss, 256, 0, c->stream>>>(c->Y, X, Xt, c->G[3], c->loss_part, c->P);
    CLAUNCH(c);
    if ((s = wgrad<32, 16>(c, 3)) || (s = conv<16, 32, BWD>(c, c->G[3], c->wp.wb[3], nullptr, c->G[2], c->A[3])) ||
        (s = wgrad<32, 32>(c, 2)) || (s = conv<32, 32, BWD>(c, c->G[2], c->wp.wb[2], nullptr, c->G[1], c->A[2])) ||
        (s = wgrad<32, 32>(c, 1)) || (s = conv<32, 32, BWD>(c, c->G[1], c->wp.wb[1], nullptr, c->G[0], c->A[1])) ||
        (s = wgrad<16, 32>(c, 0)))
        return s;
    return FFTLB_OK;
}

fftlb_status update(fftlb_cnn_t c, bool adam, float lr, float bc1, float bc2) {
    k_update<<<(FFTLB_CNN_NPARAMS + 31) / 32, 256, 0, c->stream>>>(c->gp, c->grad, c->loss, adam ? 1 : 0, c->prm, c->m, c->v, lr,
                                                                   bc1, bc2, c->wp);
    CLAUNCH(c);
    return FFTLB_OK;
}

fftlb_status check_norm(fftlb_cnn_t c, const fftlb_cnn_norm *nm, double T_run) {
    if (!nm) return fail(c, FFTLB_ERR_ARG, "NULL norm");
    if (!(nm->rho_c > 0) || !(nm->T_c > 0) || !(nm->s_rho > 0) || !(nm->s_T > 0) || !(T_run > 0))
        return fail(c, FFTLB_ERR_ARG, "norm constants and T_run must be > 0");
    return FFTLB_OK;
}

fftlb_status encode_from(fftlb_cnn_t c, fftlb_t h, double T_run, const fftlb_cnn_norm *nm, float *X) {
    fftlb::Engine *e = fftlb::engine_of(h);
    if (!e) return fail(c, FFTLB_ERR_ARG, "NULL handle");
    if (e->params().nx != c->W || e->params().ny != c->H)
        return fail(c, FFTLB_ERR_ARG, "handle grid differs from the network's grid");
    fftlb_status s = check_norm(c, nm, T_run);
    if (s != FFTLB_OK) return s;
    double *rho = c->fields, *ux = rho + c->P, *uy = ux + c->P, *T = uy + c->P;
    fftlb::Status st = e->fields(rho, ux, uy, T, true);
    if (!st.good()) return fail(c, st.code, st.msg);
    // the engine works on its own stream: order ours after it
    CCU(c, cudaStreamSynchronize(e->stream()));
    k_encode<<<grid1d(c->P), 256, 0, c->stream>>>(rho, T, X, c->P, nm->rho_c, nm->T_c, nm->s_rho, nm->s_T, T_run);
    CLAUNCH(c);
    return FFTLB_OK;
}

}  // namespace

extern "C" {

fftlb_status fftlb_cnn_create(fftlb_cnn_t *out, int H, int W, void *cuda_stream) {
    if (!out) return fail(nullptr, FFTLB_ERR_ARG, "fftlb_cnn_create: out is NULL");
    *out = nullptr;
    if (H < 1 || W < TX || W > 4096 || W % TX != 0 || H > 4096)
        return fail(nullptr, FFTLB_ERR_ARG, "grid must have 1 <= H <= 4096 and W a multiple of 64 in [64, 4096]");
    fftlb_cnn_t c = new (std::nothrow) fftlb_cnn_s();
    if (!c) return fail(nullptr, FFTLB_ERR_OOM, "host allocation failed");
    c->H = H;
    c->W = W;
    c->P = (size_t)H * W;
    c->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    auto bad = [&](fftlb_status s) {
        const std::string m = c->err;
        release(c);
        delete c;
        return fail(nullptr, s, m);
    };
    const size_t P = c->P;
    fftlb_status s = FFTLB_OK;
    if ((s = dalloc(c, &c->prm, FFTLB_CNN_NPARAMS)) || (s = dalloc(c, &c->m, FFTLB_CNN_NPARAMS)) ||
        (s = dalloc(c, &c->v, FFTLB_CNN_NPARAMS)) || (s = dalloc(c, &c->grad, FFTLB_CNN_NPARAMS)) ||
        (s = dalloc(c, &c->X, 3 * P)) || (s = dalloc(c, &c->Xt, 2 * P)) || (s = dalloc(c, &c->Y, 2 * P)) ||
        (s = dalloc(c, &c->A[0], 16 * P)) || (s = dalloc(c, &c->A[1], 32 * P)) || (s = dalloc(c, &c->A[2], 32 * P)) ||
        (s = dalloc(c, &c->A[3], 32 * P)) || (s = dalloc(c, &c->G[0], 32 * P)) || (s = dalloc(c, &c->G[1], 32 * P)) ||
        (s = dalloc(c, &c->G[2], 32 * P)) || (s = dalloc(c, &c->G[3], 16 * P)) || (s = dalloc(c, &c->loss, 1)) ||
        (s = dalloc(c, &c->fields, 4 * P)))
        return bad(s);
    for (int l = 0; l < NL; ++l) {
        if ((s = dalloc(c, &c->wp.wf[l], (size_t)9 * COUTP(l) * CINP(l))) || (s = dalloc(c, &c->wp.bias[l], COUTP(l))))
            return bad(s);
        c->wp.wb[l] = nullptr;
        if (l > 0 && (s = dalloc(c, &c->wp.wb[l], (size_t)9 * CIN_R(l) * GCH(l)))) return bad(s);
    }
    if (cudaMemset(c->prm, 0, FFTLB_CNN_NPARAMS * sizeof(float)) != cudaSuccess ||
        cudaMemset(c->m, 0, FFTLB_CNN_NPARAMS * sizeof(float)) != cudaSuccess ||
        cudaMemset(c->v, 0, FFTLB_CNN_NPARAMS * sizeof(float)) != cudaSuccess ||
        cudaMemset(c->G[3], 0, 16 * P * sizeof(bf16)) != cudaSuccess) {
        c->err = "cudaMemset failed";
        return bad(FFTLB_ERR_CUDA);
    }
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int ntiles = (H + RT - 1) / RT * (W / TX);
    c->grid_conv = std::max(1, std::min(ntiles, 2 * nsm));
    c->grid_wgrad = std::max(1, std::min(ntiles, nsm));
    c->grid_loss = std::max(1, std::min<int>((int)((P + 255) / 256), 4 * nsm));
    {
        const int wgn[NL] = {wg_size<16, 32>(), wg_size<32, 32>(), wg_size<32, 32>(), wg_size<32, 16>()};
        size_t off = 0;
        for (int l = 0; l < NL; ++l) {
            c->gp.off[l] = off;
            c->gp.wgn[l] = wgn[l];
            off += (size_t)wgn[l] * c->grid_wgrad;
        }
        if ((s = dalloc(c, &c->ws, off)) || (s = dalloc(c, &c->loss_part, c->grid_loss))) return bad(s);
        c->gp.ws = c->ws;
        c->gp.nblk = c->grid_wgrad;
        c->gp.loss_part = c->loss_part;
        c->gp.nloss = c->grid_loss;
    }
    // (per-function, process-wide: every object sets the same values)
    auto smem = [](const void *k, size_t b) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b); };
    if (smem((const void *)k_conv<16, 32, FWD_RELU>, conv_smem<16, 32>()) != cudaSuccess ||
        smem((const void *)k_conv<32, 32, FWD_RELU>, conv_smem<32, 32>()) != cudaSuccess ||
        smem((const void *)k_conv<32, 8, FWD_LAST>, conv_smem<32, 8>()) != cudaSuccess ||
        smem((const void *)k_conv<16, 32, BWD>, conv_smem<16, 32>()) != cudaSuccess ||
        smem((const void *)k_conv<32, 32, BWD>, conv_smem<32, 32>()) != cudaSuccess ||
        smem((const void *)k_wgrad<32, 16>, wgrad_smem<32, 16>()) != cudaSuccess ||
        smem((const void *)k_wgrad<32, 32>, wgrad_smem<32, 32>()) != cudaSuccess ||
        smem((const void *)k_wgrad<16, 32>, wgrad_smem<16, 32>()) != cudaSuccess) {
        c->err = "cudaFuncSetAttribute failed";
        return bad(FFTLB_ERR_CUDA);
    }
    if ((s = refresh_weights(c)) != FFTLB_OK) return bad(s);
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) {
        c->err = "initial weight tiles failed";
        return bad(FFTLB_ERR_CUDA);
    }
    *out = c;
    return FFTLB_OK;
}

fftlb_status fftlb_cnn_destroy(fftlb_cnn_t c) {
    if (!c) return FFTLB_OK;
    cudaStreamSynchronize(c->stream);
    release(c);
    delete c;
    return FFTLB_OK;
}

const char *fftlb_cnn_last_error(fftlb_cnn_t c) { return c ? c->err.c_str() : fftlb_last_error(nullptr); }

fftlb_status fftlb_cnn_set_params(fftlb_cnn_t c, const float *params, int reset_optimizer) {
    if (!c || !params) return fail(c, FFTLB_ERR_ARG, "NULL argument");
    CCU(c, cudaMemcpyAsync(c->prm, params, FFTLB_CNN_NPARAMS * sizeof(float), cudaMemcpyHostToDevice, c->stream));
    if (reset_optimizer) {
        CCU(c, cudaMemsetAsync(c->m, 0, FFTLB_CNN_NPARAMS * sizeof(float), c->stream));
        CCU(c, cudaMemsetAsync(c->v, 0, FFTLB_CNN_NPARAMS * sizeof(float), c->stream));
        c->adam_k = 0;
    }
    fftlb_status s = refresh_weights(c);
    if (s != FFTLB_OK) return s;
    CCU(c, cudaStreamSynchronize(c->stream));
    return FFTLB_OK;
}

fftlb_status fftlb_cnn_get_params(fftlb_cnn_t c, float *params) {
    if (!c || !params) return fail(c, FFTLB_ERR_ARG, "NULL argument");
    CCU(c, cudaMemcpyAsync(params, c->prm, FFTLB_CNN_NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
    CCU(c, cudaStreamSynchronize(c->stream));
    return FFTLB_OK;
}

fftlb_status fftlb_cnn_forward(fftlb_cnn_t c, const float *X, float *Y, int on_device) {
    if (!c || !Y) return fail(c, FFTLB_ERR_ARG, "NULL argument");
    c->launches = 0;
    const float *Xd = nullptr;
    fftlb_status s = upload(c, c->X, X, 3 * c->P, on_device, &Xd);
    if (s != FFTLB_OK || (s = forward(c, Xd, on_device ? Y : c->Y)) != FFTLB_OK || on_device) return s;
    CCU(c, cudaMemcpyAsync(Y, c->Y, 2 * c->P * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
    CCU(c, cudaStreamSynchronize(c->stream));
    return FFTLB_OK;
}

fftlb_status fftlb_cnn_gradient(fftlb_cnn_t c, const float *X, const float *Xt, float *grad, double *loss,
                                int on_device) {
    if (!c) return fail(c, FFTLB_ERR_ARG, "NULL network");
    c->launches = 0;
    const float *Xd = nullptr, *Xtd = nullptr;
    fftlb_status s = upload(c, c->X, X, 3 * c->P, on_device, &Xd);
    if (s != FFTLB_OK || (s = upload(c, c->Xt, Xt, 2 * c->P, on_device, &Xtd)) != FFTLB_OK ||
        (s = backward(c, Xd, Xtd)) != FFTLB_OK || (s = update(c, false, 0.f, 1.f, 1.f)) != FFTLB_OK)
        return s;
    if (grad)
        CCU(c, cudaMemcpyAsync(grad, c->grad, FFTLB_CNN_NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
    if (loss) CCU(c, cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    CCU(c, cudaStreamSynchronize(c->stream));
    return FFTLB_OK;
}

fftlb_status fftlb_cnn_train_step(fftlb_cnn_t c, const float *X, const float *Xt, float lr, double *loss,
                                  int on_device) {
    if (!c) return fail(c, FFTLB_ERR_ARG, "NULL network");
    if (!(lr > 0)) return fail(c, FFTLB_ERR_ARG, "lr must be > 0");
    c->launches = 0;
    const float *Xd = nullptr, *Xtd = nullptr;
    fftlb_status s = upload(c, c->X, X, 3 * c->P, on_device, &Xd);
    if (s != FFTLB_OK || (s = upload(c, c->Xt, Xt, 2 * c->P, on_device, &Xtd)) != FFTLB_OK ||
        (s = backward(c, Xd, Xtd)) != FFTLB_OK)
        return s;
    ++c->adam_k;
    const float bc1 = 1.f - (float)std::pow(0.9, c->adam_k), bc2 = 1.f - (float)std::pow(0.999, c->adam_k);
    if ((s = update(c, true, lr, bc1, bc2)) != FFTLB_OK) return s;
    if (loss) {
        CCU(c, cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        CCU(c, cudaStreamSynchronize(c->stream));
    }
    return FFTLB_OK;
}

fftlb_status fftlb_cnn_encode(fftlb_cnn_t c, fftlb_t h, double T_run, const fftlb_cnn_norm *norm, float *X_dev) {
    if (!c || !X_dev) return fail(c, FFTLB_ERR_ARG, "NULL argument");
    return encode_from(c, h, T_run, norm, X_dev);
}

fftlb_status fftlb_cnn_warm_start(fftlb_cnn_t c, fftlb_t h, double T_run, const fftlb_cnn_norm *norm) {
    if (!c) return fail(c, FFTLB_ERR_ARG, "NULL network");
    c->launches = 0;
    fftlb_status s = encode_from(c, h, T_run, norm, c->X);
    if (s != FFTLB_OK || (s = forward(c, c->X, c->Y)) != FFTLB_OK) return s;
    double *rho = c->fields, *u = rho + c->P, *T = u + c->P;
    k_decode<<<grid1d(c->P), 256, 0, c->stream>>>(c->X, c->Y, rho, u, T, c->P, norm->rho_c, norm->s_rho, norm->s_T,
                                                  T_run);
    CLAUNCH(c);
    CCU(c, cudaStreamSynchronize(c->stream));
    fftlb::Engine *e = fftlb::engine_of(h);
    const long steps = e->steps();
    fftlb::Status st = e->set_fields(rho, u, u, T, true);
    if (!st.good()) return fail(c, st.code, st.msg);
    e->set_steps(steps);
    return FFTLB_OK;
}

long fftlb_cnn_launches(fftlb_cnn_t c) { return c ? c->launches : 0; }

}  // extern "C"

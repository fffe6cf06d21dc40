"""The transforms of the row and column kernels (kernels_row.cuh: row_fft,
row_post, row_pre, row_dx; kernels_col.cuh: col_pass) run on the host at every
length and in both precisions: against sums written out, and without a store
outside their buffer.

Bound: an FFT of n points in arithmetic of unit roundoff u has a relative
error in the 2-norm of at most about 7 u log2 n (Higham, Accuracy and
Stability of Numerical Algorithms, Theorem 24.2); 8 u log2 n a transform, and
as much again for the products around it."""
import numpy as np

from host_device import run

PROGRAM = r"""
#include <cstdio>
#include "kernels_row.cuh"
#include "kernels_col.cuh"
using namespace fftlb;
using rk::Row;
typedef long double L;
struct Z { L x, y; };
static const L TAU = 6.283185307179586476925286766559005768L;
static Z w(long k, long n) { k %= n; return {cosl(TAU * k / n), -sinl(TAU * k / n)}; }   // exp(-2 pi i k / n)
static Z mul(Z a, Z b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
static std::vector<Z> dft(const std::vector<Z> &x, int dir) {   // (dir -1: forward)
    const int n = (int)x.size();
    std::vector<Z> t(n), o(n);
    for (int k = 0; k < n; ++k) { t[k] = w(k, n); if (dir > 0) t[k].y = -t[k].y; }
    for (int k = 0; k < n; ++k) {
        Z s{0, 0};
        for (int m = 0; m < n; ++m) { const Z p = mul(x[m], t[(long)m * k % n]); s.x += p.x; s.y += p.y; }
        o[k] = s;
    }
    return o;
}
static unsigned seed = 1;
static double rnd() { seed = seed * 1664525u + 1013904223u; return (seed >> 8) / 8388608.0 - 1.0; }
template <typename C> static double err(const C *a, const std::vector<Z> &b) {   // relative, 2-norm
    L e = 0, s = 0;
    for (size_t i = 0; i < b.size(); ++i) {
        const L dx = a[i].x - b[i].x, dy = a[i].y - b[i].y;
        e += dx * dx + dy * dy;
        s += b[i].x * b[i].x + b[i].y * b[i].y;
    }
    return (double)sqrtl(e / s);
}
constexpr int PAD = 64;   // values around a buffer that nothing may touch
template <typename C> struct Buffer {
    std::vector<C> v;
    size_t n;
    Buffer(size_t n_) : v(n_ + 2 * PAD, C{77, 77}), n(n_) {}
    C *p() { return v.data() + PAD; }
    bool kept() const {
        for (int i = 0; i < PAD; ++i)
            if (v[i].x != 77 || v[i].y != 77 || v[PAD + n + i].x != 77 || v[PAD + n + i].y != 77) return false;
        return true;
    }
};
template <typename real, int H> void rows() {
    using C = typename cplx_of<real>::type;
    constexpr int P = Row<real, H>::P, E = H / P;
    std::vector<C> tw(H), wh(H / 2), wp(H / 2);
    for (int k1 = 0; k1 < E; ++k1)
        for (int l = 0; l < P; ++l) { const Z a = w((long)l * k1, H); tw[k1 * P + l] = C{(real)a.x, (real)a.y}; }
    std::vector<real> kx(H);
    for (int k = 0; k < H; ++k) kx[k] = (real)rnd();
    for (int k = 0; k < H / 2; ++k) {
        const Z a = w(k, 2 * H);
        wp[k] = C{(real)a.x, (real)a.y};
        wh[k] = C{(real)(a.x / 2), (real)(a.y / 2)};
    }
    std::vector<Z> x(H);
    for (auto &z : x) z = {(L)(real)rnd(), (L)(real)rnd()};
    auto fill = [&](Buffer<C> &b) { for (int i = 0; i < H; ++i) b.p()[i] = C{(real)x[i].x, (real)x[i].y}; };
    Buffer<C> f(H), g(H), X(H), y(H), d(H);
    fill(f); fill(g); fill(d);
    run_block(P, [&] { rk::row_fft<H, -1>(f.p(), tw.data(), (int)threadIdx.x); });
    run_block(P, [&] { rk::row_fft<H, +1>(g.p(), tw.data(), (int)threadIdx.x); });
    const double e0 = err(f.p(), dft(x, -1)), e1 = err(g.p(), dft(x, +1));
    // the real row x[2m] + i x[2m + 1]: its one-sided spectrum, packed
    std::vector<Z> r(2 * H), R(H);
    for (int m = 0; m < H; ++m) { r[2 * m] = {x[m].x, 0}; r[2 * m + 1] = {x[m].y, 0}; }
    const std::vector<Z> full = dft(r, -1);
    for (int k = 0; k < H; ++k) R[k] = k ? full[k] : Z{full[0].x, full[H].x};
    run_block(P, [&] { rk::row_post<H>(f.p(), wh.data(), (int)threadIdx.x, [&](int k, C v) { X.p()[k] = v; }); });
    const double e2 = err(X.p(), R);
    // and back, times 2 H
    run_block(P, [&] {
        rk::row_pre<H, 1>(y.p(), wp.data(), (int)threadIdx.x, X.p(), X.p(), [](int, C a, C) { return a; }, [] {});
        __syncwarp();
        rk::row_fft<H, +1>(y.p(), tw.data(), (int)threadIdx.x);
    });
    std::vector<Z> back(H);
    for (int m = 0; m < H; ++m) back[m] = {x[m].x * 2 * H, x[m].y * 2 * H};
    const double e3 = err(y.p(), back);
    // i k_x X / 2H, DC and Nyquist zero
    run_block(P, [&] {
        rk::row_fft<H, -1>(d.p(), tw.data(), (int)threadIdx.x);
        rk::row_dx<H>(d.p(), wh.data(), wp.data(), kx.data(), (int)threadIdx.x);
        __syncwarp();
        rk::row_fft<H, +1>(d.p(), tw.data(), (int)threadIdx.x);
    });
    std::vector<Z> D(2 * H), dd(H);
    for (int k = 1; k < H; ++k) {
        const L m = (L)kx[k] / (2 * H);
        D[k] = {-m * full[k].y, m * full[k].x};
        D[2 * H - k] = {D[k].x, -D[k].y};
    }
    const std::vector<Z> dr = dft(D, +1);
    for (int m = 0; m < H; ++m) dd[m] = {dr[2 * m].x, dr[2 * m + 1].x};
    const double e4 = err(d.p(), dd);
    const bool kept = f.kept() && g.kept() && X.kept() && y.kept() && d.kept();
    std::printf("row %d %d %d %.3e %.3e %.3e %.3e %.3e\n", (int)sizeof(real), H, kept, e0, e1, e2, e3, e4);
}
template <typename real, int NY> void cols() {
    using G = ck::Col<real, NY>;
    using C = typename G::C;
    constexpr int P = G::P, E = G::E, TW = G::TW;
    // the tile, with the tables behind it as the kernels find them, or elsewhere
    std::vector<C> tab(2 * NY + P + NY / 2 + 1);
    for (int k1 = 0; k1 < E; ++k1)
        for (int l = 0; l < P; ++l) {
            const Z a = w((long)l * k1, NY);
            tab[k1 * P + l] = tab[NY + l * E + k1] = C{(real)a.x, (real)a.y};
        }
    for (int k = 0; k < P; ++k) { const Z a = w(k, P); tab[2 * NY + k] = C{(real)a.x, (real)a.y}; }
    Buffer<C> T((size_t)NY * TW + (G::TABS ? tab.size() : 0));
    if (G::TABS) std::copy(tab.begin(), tab.end(), T.p() + (size_t)NY * TW);
    const ck::ColTab<real, NY> tb(T.p(), tab.data());
    std::vector<Z> m(NY);
    for (auto &z : m) z = {(L)(real)rnd(), (L)(real)rnd()};
    std::vector<C> in((size_t)NY * TW), out((size_t)NY * TW), X((size_t)NY * TW);
    for (auto &z : in) z = C{(real)rnd(), (real)rnd()};
    std::vector<int> seen((size_t)NY * TW, 0);
    uint64_t bar = 0;
    int e = 0;
    for (int inv = 0; inv < 2; ++inv)
        run_block(G::NT, [&] {
            const int c = threadIdx.x % TW, jl = threadIdx.x / TW;
            C v[E];
            for (int q = 0; q < E; ++q) v[q] = in[(size_t)(jl + P * q) * TW + c];
            auto mult = [&](int k, C u) {
                X[(size_t)k * TW + c] = u;
                ++seen[(size_t)k * TW + c];
                return C{(real)(u.x * m[k].x - u.y * m[k].y), (real)(u.x * m[k].y + u.y * m[k].x)};
            };
            if (inv) {
                ck::col_pass<real, NY, true>(v, T.p(), tb, &bar, &e, c, jl, mult);
                for (int q = 0; q < E; ++q) out[(size_t)(jl + P * q) * TW + c] = v[q];
            } else {
                ck::col_pass<real, NY, false>(v, T.p(), tb, &bar, &e, c, jl, mult);
            }
        });
    double e0 = 0, e1 = 0;
    bool once = true;
    for (int s : seen) once = once && s == 2;   // (one per pass)
    for (int c = 0; c < TW; c += TW - 1) {
        std::vector<Z> x(NY);
        std::vector<C> a(NY), b(NY);
        for (int k = 0; k < NY; ++k) {
            x[k] = {in[(size_t)k * TW + c].x, in[(size_t)k * TW + c].y};
            a[k] = X[(size_t)k * TW + c];
            b[k] = out[(size_t)k * TW + c];
        }
        std::vector<Z> f = dft(x, -1);
        e0 = std::fmax(e0, err(a.data(), f));
        for (int k = 0; k < NY; ++k) f[k] = mul(f[k], m[k]);
        e1 = std::fmax(e1, err(b.data(), dft(f, +1)));
    }
    std::printf("col %d %d %d %.3e %.3e\n", (int)sizeof(real), NY, T.kept() && once, e0, e1);
}
template <typename real, int... H> void all_rows() { (rows<real, H>(), ...); }
template <typename real, int... N> void all_cols() { (cols<real, N>(), ...); }
int main() {
    all_rows<float, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024>();
    all_rows<double, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512>();
    all_cols<float, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048>();
    all_cols<double, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024>();
}
"""


def test_transforms_of_the_row_and_column_kernels(tmp_path):
    lines = run(tmp_path, PROGRAM)
    assert len(lines) == 13 + 11 + 15 + 13
    for kind, *v in lines:
        size, n, kept, *errs = map(float, v)
        u = 2.0 ** -24 if size == 4 else 2.0 ** -53
        one = 8 * u * np.log2(2 * n if kind == "row" else n)
        # a transform; a transform and the pass to or from real rows; two transforms
        bounds = [one, one, 2 * one, 4 * one, 4 * one] if kind == "row" else [one, 3 * one]
        assert kept, (kind, v)
        assert all(e <= b for e, b in zip(errs, bounds)), (kind, v, bounds)

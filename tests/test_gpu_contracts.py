"""What the C ABI promises about its buffers, its batches, its rounding and its
tuning, where a fast route could break it."""
import numpy as np
import pytest

from gpu_common import lib
from oracle import fftlb_oracle as O
from paper_1011_3582_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fl():
    return lib()


def gradient_of(h, g, n, shape):
    """The gradient of n fields between disjoint, aligned buffers."""
    out = torch.empty((2 * n,) + shape, dtype=torch.float64, device="cuda")
    h.gradient(g, out, n)
    torch.cuda.synchronize()
    return out


# two routes, each within 1e-12 (fp64) or 2e-5 (fp32) of the largest derivative
# from the true one (test_gpu_spectral.py)
GRADIENT_TOL = {64: 2e-12, 32: 4e-5}


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx,ny", [(64, 64), (32, 12), (96, 24), (36, 16)])
@pytest.mark.parametrize("n,at", [(1, 0), (1, 1), (3, 0), (3, 2), (2, 0.5)])
def test_gradient_output_may_overlap_its_input(fl, nx, ny, precision, n, at):
    """g lies in out's range, from plane `at` of it on (the last case: half a
    plane in); every derivative is that of the g handed over."""
    rng = np.random.default_rng(nx + ny + n)
    src = torch.from_numpy(rng.standard_normal((n, ny, nx))).cuda()
    with fl.Handle(fl.params(nx=nx, ny=ny, precision=precision)) as h:
        ref = gradient_of(h, src, n, (ny, nx))
        buf = torch.empty(2 * n * ny * nx, dtype=torch.float64, device="cuda")
        first = int(at * ny * nx)
        g = buf[first:first + n * ny * nx].view(n, ny, nx)
        g.copy_(src)
        torch.cuda.synchronize()
        h.gradient(g, buf, n)
        torch.cuda.synchronize()
    err = (buf.view(2 * n, ny, nx) - ref).abs().amax(dim=(1, 2))
    assert (err <= GRADIENT_TOL[precision] * ref.abs().amax(dim=(1, 2))).all()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx,ny", [(64, 64), (32, 12), (48, 16), (36, 16)])
@pytest.mark.parametrize("goff,ooff", [(1, 0), (0, 1), (1, 1)])
def test_gradient_takes_buffers_on_any_double(fl, nx, ny, precision, goff, ooff):
    """g and out one double off a 16-byte boundary."""
    n, N = 2, nx * ny
    rng = np.random.default_rng(nx * ny + goff)
    src = torch.from_numpy(rng.standard_normal((n, ny, nx))).cuda()
    with fl.Handle(fl.params(nx=nx, ny=ny, precision=precision)) as h:
        ref = gradient_of(h, src, n, (ny, nx))
        g = torch.empty(n * N + 1, dtype=torch.float64, device="cuda")[goff:goff + n * N].view(n, ny, nx)
        buf = torch.full((2 * n * N + 2,), 7.0, dtype=torch.float64, device="cuda")
        out = buf[ooff:ooff + 2 * n * N].view(2 * n, ny, nx)
        g.copy_(src)
        torch.cuda.synchronize()
        h.gradient(g, out, n)
        torch.cuda.synchronize()
    err = (out - ref).abs().amax(dim=(1, 2))
    assert (err <= GRADIENT_TOL[precision] * ref.abs().amax(dim=(1, 2))).all()
    assert (buf[:ooff] == 7.0).all() and (buf[ooff + 2 * n * N:] == 7.0).all()


@pytest.mark.parametrize("nx,ny,runs", [(256, 256, 4), (512, 162, 2), (1024, 96, 2), (256, 648, 2), (512, 324, 2), (1024, 162, 2)])
def test_fp32_batch_runs_equal_single_handles_at_any_group_size(fl, nx, ny, runs):
    """A run's bits do not depend on how many runs share its group: three shapes that
    alone have too few rows for the persistent row kernels, and three that have
    enough."""
    prm = fl.params(nx=nx, ny=ny, integrator=3, precision=32)
    starts = [W.smooth_random(nx, ny, seed=s, rho0=1.3, T0=0.9, amp=0.05, umax=0.02) for s in range(runs)]
    with fl.Batch([prm] * runs, autotune=False) as b:
        for i, f in enumerate(starts):
            b.set_fields(i, *f)
        b.step(2)
        got = [(b.get_f(i), b.invariants(i)) for i in range(runs)]
    for f, (g, inv) in zip(starts, got):
        with fl.Handle(prm) as h:
            h.set_fields(*f)
            h.step(2)
            assert np.array_equal(h.get_f(), g)
            assert h.invariants() == inv


@pytest.mark.parametrize("nx,ny,nstates", [(64, 32, 24), (256, 16, 12), (1024, 96, 12), (36, 16, 12)])
def test_fp32_relaxation_is_rounded_after_the_difference(fl, nx, ny, nstates):
    """One Euler step of a uniform state: no derivative term, so f' = f - (dt /
    tau) (f - f^eq).  A handle with dt = tau = 1 returns the kernel's own f^eq
    (f - (f - f^eq) is exact for neighbouring numbers).  With dt = tau = 0.01
    the result is the same sum with 1 / tau and dt rounded: (f - f^eq), below
    2^-16 of f here, is exact or rounded once, the products after it carry three
    roundings of that small number, and the last addition rounds f' itself, by
    at most u = 2^-24 of it: together below (1 + 2^-10) u.  Two products of the
    size of f / tau, subtracted, would each leave a rounding of their own."""
    rng = np.random.default_rng(nx + ny)
    one = np.ones((ny, nx))
    worst = 0.0
    with fl.Handle(fl.params(nx=nx, ny=ny, integrator=1, precision=32, dt=1.0, tau=1.0)) as h1, \
            fl.Handle(fl.params(nx=nx, ny=ny, integrator=1, precision=32, dt=0.01, tau=0.01)) as h:
        for _ in range(nstates):
            rho, T = rng.uniform(0.4, 1.6), rng.uniform(0.85, 1.0)
            ux, uy = rng.uniform(-0.05, 0.05, 2)
            h1.set_fields(rho * one, ux * one, uy * one, T * one)
            f = h1.get_f()[:, 0, 0]
            h1.step(1)
            feq = h1.get_f()[:, 0, 0]
            assert (np.abs(f - feq) < 2.0 ** -16 * np.abs(f)).all()
            h.set_fields(rho * one, ux * one, uy * one, T * one)
            h.step(1)
            got = h.get_f()
            assert (got == got[:, :1, :1]).all()
            r = float(np.float32(0.01)) / float(np.float32(0.01))
            want = f + r * (feq - f)
            worst = max(worst, (np.abs(got[:, 0, 0] - want) / np.abs(want)).max())
    assert worst <= (1 + 2.0 ** -10) * 2.0 ** -24


@pytest.mark.parametrize("nx,ny,tuned", [(128, 64, ()), (36, 64, (2, 3, 4)), (64, 54, (0, 1)), (36, 54, (0, 1, 2, 3, 4))])
def test_autotune_times_only_what_the_stage_launches(fl, nx, ny, tuned):
    """A grid whose rows and columns take no runtime parameter is timed once (two
    warm-up stages and three timed ones) and keeps its parameters; with one axis
    on the pipelined kernels only that axis's parameters move."""
    f = W.smooth_random(nx, ny, seed=3, rho0=1.3, T0=0.9, amp=0.05, umax=0.02)
    with fl.Handle(fl.params(nx=nx, ny=ny, precision=32)) as h:
        h.set_fields(*f)
        before, f0 = h.tuning(), h.get_f()
        h.profile(True)
        ms = h.autotune()
        stages = h.profile_read()["row_forward_moments"][1]
        h.profile(False)
        after = h.tuning()
        assert ms > 0 and np.array_equal(h.get_f(), f0)
    assert (stages == 5) == (not tuned)
    assert all(a == b for i, (a, b) in enumerate(zip(before, after)) if i not in tuned)


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx,ny", [(36, 18), (96, 48), (384, 288), (384, 324)])
def test_invariants_on_both_sides_of_the_wide_site_sums(fl, nx, ny, precision):
    """The conservation sums with one and with four sites a thread (the last
    grid), measured against the sums of the parts' absolute values: every
    per-site value carries at most 16 roundings, summed in fp64."""
    f = W.smooth_random(nx, ny, seed=nx + ny, rho0=1.3, T0=0.9, amp=0.05, umax=0.02)
    p = O.Params(nx=nx, ny=ny)
    with fl.Handle(fl.params(nx=nx, ny=ny, precision=precision)) as h:
        h.set_fields(*f)
        inv = h.invariants()
    f0 = O.init_equilibrium(*f, p)
    ref = O.invariants(f0, p)
    rho, ux, uy, T = O.moments(f0)
    area = p.dx ** 2
    grad2 = O.D(rho, "x", p.dx, 4) ** 2 + O.D(rho, "y", p.dx, 4) ** 2
    scale = dict(mass=rho.sum() * area, px=(4.3 * rho).sum() * area, py=(4.3 * rho).sum() * area, umax=4.3,
                 eT=(rho * T + p.a * rho ** 2 + p.K * grad2 / 2 + rho).sum() * area)
    for k, s in scale.items():
        assert abs(inv[k] - ref[k]) <= (1e-13 if precision == 64 else 2e-6) * s

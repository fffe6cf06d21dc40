"""Parity of the cluster-shared row kernels and the register-loaded column
kernels (kernels_row.cuh, kernels_col.cuh) with the oracle: one SSP-RK3 step at
every row length (with a short other axis) and every column length, the two
precisions, zeta and H off zero so that every derivative row counts; odd
partners (a length that only the general kernels take) on the other axis; and
runs of one batch against single handles.

Tolerances: fp64 1e-9 relative to the largest f (the stated bar); fp32
gpu_common.fp32_force_bound, elementwise against max(|f|, mean |f|) as in the
parity tests."""
import numpy as np
import pytest

from gpu_common import fp32_force_bound, lib
from oracle import fftlb_oracle as O
from paper_1011_3582_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROWS = [32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048]
COLS = [4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048]
SHAPES = [(n, 6) for n in ROWS] + [(32, n) for n in COLS] + [(36, 64), (64, 54), (12, 96), (8, 16)]


# rows just above the line where the persistent fp32 rows take over (one row a
# block) and a few more than their resident blocks (a second row in some)
PERSISTENT = [(256, 648), (256, 1296), (512, 324), (512, 648), (1024, 162), (1024, 324)]


@pytest.fixture(scope="module")
def fl():
    return lib()


def fields_of(nx, ny, seed):
    return W.smooth_random(nx, ny, seed=seed, rho0=1.3, T0=0.9, amp=0.05, umax=0.02)


@pytest.mark.parametrize("nx,ny,precision", [(nx, ny, p) for nx, ny in SHAPES for p in (64, 32)] +
                         [(nx, ny, 32) for nx, ny in PERSISTENT])
def test_one_step_matches_oracle(fl, nx, ny, precision):
    if precision == 64 and max(nx, ny) > 1024:
        pytest.skip("fp64 grids end at 1024")
    f = fields_of(nx, ny, nx + ny)
    kw = dict(nx=nx, ny=ny, zeta=1e-3, H=1e-6, K=1e-5)
    p = O.Params(integrator=3, **kw)
    ref = O.run(O.init_equilibrium(*f, p), p, 1)
    with fl.Handle(fl.params(integrator=3, precision=precision, **kw)) as h:
        h.set_fields(*f)
        h.step(1)
        out = h.get_f()
    bound = 1e-9 if precision == 64 else fp32_force_bound((ny, nx), 1, f[0], f[3], K=1e-5 + 1e-6)
    scale = np.maximum(np.abs(ref), np.abs(ref).mean())
    assert (np.abs(out - ref) / scale).max() < bound


@pytest.mark.parametrize("precision", [64, 32])
def test_batch_runs_equal_single_handles(fl, precision):
    """Three runs of one shape in one launch give each run's own result."""
    nx, ny = 96, 12
    prm = fl.params(nx=nx, ny=ny, integrator=3, precision=precision)
    starts = [fields_of(nx, ny, s) for s in (1, 2, 3)]
    with fl.Batch([prm] * 3, autotune=False) as b:
        for i, f in enumerate(starts):
            b.set_fields(i, *f)
        b.step(2)
        got = [(b.get_f(i), b.invariants(i)) for i in range(3)]
    for f, (g, inv) in zip(starts, got):
        with fl.Handle(prm) as h:
            h.set_fields(*f)
            h.step(2)
            assert np.array_equal(h.get_f(), g)
            assert h.invariants() == inv


@pytest.mark.parametrize("nx,ny", [(64, 64), (192, 48), (512, 512), (36, 36)])
def test_uniform_state_is_a_bitwise_fixed_point_in_fp32(fl, nx, ny):
    """On a uniform state at rest a stage changes f by rounding noise alone:
    (f - f^eq) dt / tau is a few u = 2^-24 times 1e-3, and the convection of a
    uniform row the transforms' round-off, below v k_max u dt = 4.3 * 660 *
    1e-5 u = 0.03 u, of f.  Both are below half an ulp (at least u / 2 of f), so
    the Runge-Kutta combination, which adds a small increment to the base
    state, returns the state bit for bit.  (Weighting f^n and f^1 by fp32's 1/3
    and 2/3, which add up to 1 + 3e-8, would scale it every step.)"""
    rho, u, T = 1.1, np.zeros((ny, nx)), 0.9
    with fl.Handle(fl.params(nx=nx, ny=ny, integrator=3, precision=32)) as h:
        h.set_fields(np.full((ny, nx), rho), u, u.copy(), np.full((ny, nx), T))
        f0 = h.get_f()
        h.step(20)
        assert np.array_equal(h.get_f(), f0)


GRAD = [(n, 6) for n in ROWS] + [(32, n) for n in COLS]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx,ny", GRAD)
def test_gradient_and_invariants_match_oracle(fl, nx, ny, precision):
    """fftlb_gradient of three fields (bounds of test_gpu_spectral.py: 1e-12 and
    2e-5 of the largest derivative) and the conservation sums of a state: every
    per-site value carries at most 16 roundings (2e-15, 1e-6 relative), summed
    in fp64, measured against the sums of the parts' absolute values."""
    if precision == 64 and max(nx, ny) > 1024:
        pytest.skip("fp64 grids end at 1024")
    rng = np.random.default_rng(nx * 7 + ny)
    g = rng.standard_normal((3, ny, nx))
    f = fields_of(nx, ny, nx + 2 * ny)
    p = O.Params(nx=nx, ny=ny)
    with fl.Handle(fl.params(nx=nx, ny=ny, precision=precision)) as h:
        gd = torch.from_numpy(g).cuda()
        out = torch.empty((6, ny, nx), dtype=torch.float64, device="cuda")
        h.gradient(gd, out, 3)
        torch.cuda.synchronize()
        h.set_fields(*f)
        inv = h.invariants()
    out = out.cpu().numpy()
    tol = 1e-12 if precision == 64 else 2e-5
    for i in range(3):
        for q, ax in ((0, "x"), (1, "y")):
            d = O.D(g[i], ax, 1 / 256, 4)
            assert np.abs(out[2 * i + q] - d).max() <= tol * np.abs(d).max()
    f0 = O.init_equilibrium(*f, p)
    ref = O.invariants(f0, p)
    rho, ux, uy, T = O.moments(f0)
    area = p.dx ** 2
    grad2 = O.D(rho, "x", p.dx, 4) ** 2 + O.D(rho, "y", p.dx, 4) ** 2
    scale = dict(mass=rho.sum() * area, px=(4.3 * rho).sum() * area, py=(4.3 * rho).sum() * area, umax=4.3,
                 eT=(rho * T + p.a * rho ** 2 + p.K * grad2 / 2 + rho).sum() * area)
    for k, s in scale.items():
        assert abs(inv[k] - ref[k]) <= (1e-13 if precision == 64 else 2e-6) * s


@pytest.mark.parametrize("precision", [64, 32])
def test_device_reads_into_unaligned_buffers(fl, precision):
    """Device buffers one value off 16-byte alignment take the scalar accesses
    and give the same values, in and out."""
    nx, ny = 36, 18
    n = nx * ny
    f = fields_of(nx, ny, 5)
    with fl.Handle(fl.params(nx=nx, ny=ny, precision=precision)) as h:
        h.set_fields(*f)
        buf = torch.empty(33 * n + 1, dtype=torch.float64, device="cuda")
        off = buf[1:].view(33, ny, nx)
        h.get_f(off, on_device=True)
        ref = torch.empty((33, ny, nx), dtype=torch.float64, device="cuda")
        h.get_f(ref, on_device=True)
        fo = [torch.empty(n + 1, dtype=torch.float64, device="cuda")[1:].view(ny, nx) for _ in range(4)]
        h.fields(*fo, on_device=True)
        host = h.fields()
        torch.cuda.synchronize()
        assert torch.equal(off, ref)
        for a, b in zip(fo, host):
            assert np.array_equal(a.cpu().numpy(), b)
        h.set_f(off, on_device=True)
        assert np.array_equal(h.get_f(), ref.cpu().numpy())

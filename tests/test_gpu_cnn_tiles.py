"""The warm-start network's kernels at the edges of their 64-pixel x 4-row
tiles (ragged heights, one row, several tiles a row) against the oracle with
the same bfloat16 rounding points, with the bounds of test_gpu_warmstart.py;
a gradient is the same bits on every call (no atomics)."""
import numpy as np
import pytest

from gpu_common import lib
from oracle import cnn_oracle as C
from test_gpu_warmstart import U, bf16_params, case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fl():
    return lib()


@pytest.mark.parametrize("H,Wd", [(1, 64), (2, 64), (3, 128), (5, 64), (9, 192)])
def test_tile_edges(fl, H, Wd):
    params, X, Xt = case(H + Wd, H, Wd)
    p32 = bf16_params(fl, params)
    with fl.CNN(H, Wd) as net:
        net.set_params(fl.pack_params(params))
        Y = net.forward(X)
        loss, g = net.gradient(X, Xt)
        loss2, g2 = net.gradient(X, Xt)
    assert loss == loss2 and np.array_equal(g, g2)
    Yr, _ = C.forward(p32, X, bf16=True)
    err = np.abs(Y - Yr)
    assert err.max() <= 4 * U * np.abs(Yr).max() and err.mean() <= 0.05 * U * np.abs(Yr).max()
    L_ref, grads = C.loss_and_grads(p32, X, Xt, bf16=True)
    assert loss == pytest.approx(L_ref, rel=1e-4)
    o = 0
    for pair in grads:
        for arr in pair:
            a, b = g[o:o + arr.size].astype(np.float64), np.asarray(arr, np.float64).ravel()
            assert np.linalg.norm(a - b) <= 2 * U * np.linalg.norm(b)
            o += arr.size

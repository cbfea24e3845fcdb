"""The network's kernel at the edges of its 32-sample tiles and of its grid
(one sample, a ragged last tile, more tiles than blocks), against the float64
oracle with the tolerances of test_gpu_mlp.py, and deterministic."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    engine()
    from paper_1204_5072_gb300 import surrogate
    return surrogate


@pytest.mark.parametrize("n", [1, 31, 32, 33, 129, 9733, 20001])
def test_tiles(S, n):
    theta = S.init_params(n)
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, 4)).astype(np.float32)
    t = (np.sin(x[:, 0]) + 0.5 * x[:, 1] * x[:, 2] - 0.3 * x[:, 3] ** 2 + 0.2).astype(np.float32)
    m = S.MLP(theta)
    y, ref = m.predict(x), M.forward(theta, x)
    assert np.max(np.abs(y - ref)) <= 2e-4 * np.max(np.abs(ref)) + 1e-5
    loss, g = m.loss_grad(x, t)
    rl, rg = M.loss_and_grad(theta, x, t)
    assert loss == pytest.approx(rl, rel=1e-4)
    for name, _ in M.SHAPES:
        a, b = M.unflatten(g)[name].ravel(), M.unflatten(rg)[name].ravel()
        assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b) + 1e-7, name
    loss2, g2 = m.loss_grad(x, t)
    assert loss2 == loss and np.array_equal(g, g2) and np.array_equal(m.predict(x), y)
    m.close()


def test_loss_without_gradient(S):
    import ctypes
    from paper_1204_5072_gb300._lib import _ptr, load
    x = np.random.default_rng(3).standard_normal((70, 4)).astype(np.float32)
    t = x[:, 0].copy()
    m = S.MLP(S.init_params(2))
    want, _ = m.loss_grad(x, t)
    out = ctypes.c_float()
    assert load().kpz_mlp_loss_grad(m._m, _ptr(x), _ptr(t), 70, ctypes.byref(out), None) == 0
    assert out.value == want
    m.close()

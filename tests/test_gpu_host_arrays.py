"""Callers' host arrays as the C ABI takes them: any address, whether or not the
kernels could use it in place."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_5072_gb300._lib import _ptr, load
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    return engine()


def at_offset(n, dtype, offset):
    """n values whose address is `offset` bytes beyond a multiple of 64."""
    raw = np.zeros(n * np.dtype(dtype).itemsize + 128, np.uint8)
    start = -raw.ctypes.data % 64 + offset
    out = raw[start:start + n * np.dtype(dtype).itemsize].view(dtype)
    assert out.ctypes.data % 64 == offset
    return out


# 2048: several bands of the staging area.
@pytest.mark.parametrize("L", [128, 512, 2048])
@pytest.mark.parametrize("offset", [0, 8, 16, 24, 4, 1])
def test_heights(eng, L, offset):
    st = O.State.flat(L).run(3, 128, 128, 0.7, 0.4, seed=5)
    st.h00, st.t = -3, 2
    lat = eng.Lattice(L)
    lat.set_slopes(st.packed(), h00=st.h00, t=st.t)
    for absolute in (0, 1):
        out = at_offset(L * L, np.int64, offset)
        assert load().kpz_heights(lat.handle, _ptr(out), absolute) == 0
        assert np.array_equal(out.reshape(L, L), st.heights(absolute=bool(absolute)))
    lat.close()


# The network: unaligned arrays give the bits aligned ones do, and an output may
# overlap an input.
@pytest.fixture(scope="module")
def net(eng):
    from paper_1204_5072_gb300 import surrogate
    mlp = surrogate.MLP(surrogate.init_params(5))
    n = 9000
    x = np.random.default_rng(5).standard_normal((n, 4)).astype(np.float32)
    t = x[:, 0].copy()
    yield mlp, n, x, t, mlp.predict(x), mlp.loss_grad(x, t)
    mlp.close()


@pytest.mark.parametrize("ox,ot,oy", [(1, 0, 0), (0, 2, 0), (0, 0, 3), (2, 6, 1), (4, 8, 12)])
def test_network_arrays(net, ox, ot, oy):
    import ctypes
    mlp, n, x, t, y, (loss, grad) = net
    ux, ut = at_offset(4 * n, np.float32, ox), at_offset(n, np.float32, ot)
    ux[:], ut[:] = x.ravel(), t
    out = at_offset(n, np.float32, oy)
    assert load().kpz_mlp_predict(mlp._m, _ptr(ux), n, _ptr(out)) == 0
    assert np.array_equal(out, y)
    g, l = at_offset(len(grad), np.float32, oy), ctypes.c_float()
    assert load().kpz_mlp_loss_grad(mlp._m, _ptr(ux), _ptr(ut), n, ctypes.byref(l), _ptr(g)) == 0
    assert l.value == loss and np.array_equal(g, grad)
    assert np.array_equal(mlp.predict(ux.reshape(n, 4)), y)   # numpy hands an unaligned view on as it is
    assert np.array_equal(mlp.loss_grad(ux.reshape(n, 4), ut)[1], grad)


@pytest.mark.parametrize("shift", [0, 1, 4000])
def test_network_output_over_its_input(net, shift):
    import ctypes
    mlp, n, x, t, y, (loss, grad) = net
    xs = x.ravel().copy()
    assert load().kpz_mlp_predict(mlp._m, _ptr(xs), n, _ptr(xs[shift:])) == 0
    assert np.array_equal(xs[shift:shift + n], y)
    xs = x.ravel().copy()
    assert load().kpz_mlp_loss_grad(mlp._m, _ptr(xs), _ptr(t), n, ctypes.byref(ctypes.c_float()), _ptr(xs[shift // 2:])) == 0
    assert np.array_equal(xs[shift // 2:][:len(grad)], grad)
    ts = np.concatenate([t, np.zeros(len(grad), np.float32)])
    assert load().kpz_mlp_loss_grad(mlp._m, _ptr(x), _ptr(ts), n, ctypes.byref(ctypes.c_float()), _ptr(ts[shift:])) == 0
    assert np.array_equal(ts[shift:][:len(grad)], grad)


@pytest.mark.parametrize("n", [2 ** 31 - 31, 2 ** 31, 2 ** 32 - 1])
def test_network_refuses_more_samples_than_it_counts(net, n):
    """Answered from the count alone: the arrays are far smaller and stay as they are."""
    import ctypes
    from paper_1204_5072_gb300._lib import KPZ_ENOMEM
    m, lib, l = net[0]._m, load(), ctypes.c_float(-1.0)
    x, t, order = np.full(64, 7, np.float32), np.full(16, 7, np.float32), np.zeros(16, np.uint32)
    assert lib.kpz_mlp_predict(m, _ptr(x), n, _ptr(t)) == KPZ_ENOMEM
    assert lib.kpz_mlp_loss_grad(m, _ptr(x), _ptr(t), n, ctypes.byref(l), None) == KPZ_ENOMEM
    assert lib.kpz_mlp_train(m, _ptr(x), _ptr(t), 16, _ptr(order), 1, n, ctypes.c_float(1e-3), ctypes.byref(l)) == KPZ_ENOMEM
    assert l.value == -1.0 and (x == 7).all() and (t == 7).all()


def test_slopes_into_a_used_array_cost_a_copy(eng):
    """An export into an array whose pages exist takes about as long as the copy
    it is (1.3 times at this size; touching every page first made it 2.4)."""
    import time
    import torch
    L = 16384
    lat = eng.Lattice(L)
    out = np.zeros(L * L // 16, np.uint32)
    host, dev = torch.from_numpy(out.view(np.int32)), torch.zeros(L * L // 16, dtype=torch.int32, device="cuda")

    def best(f):
        times = []
        for _ in range(30):
            t = time.perf_counter()
            f()
            times.append(time.perf_counter() - t)
        return min(times)

    assert best(lambda: lat.slopes_into(out)) < 1.8 * best(lambda: host.copy_(dev))
    lat.close()

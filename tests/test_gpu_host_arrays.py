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

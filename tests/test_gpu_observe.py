"""Exact W^2 and heights at the edges of their kernels' splits: fewer block
columns than row segments, one block and many, rough, flat and steep surfaces,
odd start parity, repeated calls; host arrays small and large."""
import numpy as np
import pytest

from oracle import oracle as O
from synth import inputs as I
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    return engine()


@pytest.mark.parametrize("L", [128, 256, 512, 1024, 2048])
def test_width_and_heights(eng, L):
    states = [O.State.flat(L), O.State.flat(L).run(4, 128, 128, 0.7, 0.4, seed=5),
              O.State(L, *I.separable_surface(L, 8))]
    for k, st in enumerate(states):
        st.h00, st.t = 6 * k - 7, k
        lat = eng.Lattice(L)
        lat.set_slopes(st.packed(), h00=st.h00, t=st.t)
        for _ in range(2):
            r = lat.roughness()
            assert (r["S1"], r["S2"], r["h00"], r["w2"]) == (*st.sums(), st.h00, st.w2())
        assert np.array_equal(lat.heights(), st.heights())
        assert np.array_equal(lat.heights(absolute=True), st.heights(absolute=True))
        lat.close()


def test_largest_sums(eng):
    """A lattice with every row a tent of height L / 2: S2 near its maximum."""
    L = 4096
    sx = np.zeros((L, L), np.uint8)
    sx[:, :L // 2] = 1
    sy = np.zeros((L, L), np.uint8)
    sy[:L // 2, :] = 1
    st = O.State(L, sx, sy)
    lat = eng.Lattice(L)
    lat.set_slopes(st.packed())
    i = np.arange(L, dtype=np.int64)
    f = np.minimum(i, L - i)
    n, s, s2 = L, int(f.sum()), int((f * f).sum())
    r = lat.roughness()
    assert r["S1"] == 2 * n * s and r["S2"] == 2 * n * s2 + 2 * s * s
    assert np.array_equal(lat.heights(), f[None, :] + f[:, None])
    lat.close()

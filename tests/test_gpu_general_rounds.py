"""The general-rate rounds that run from shared memory, in the work-queue sweep
and in the batch: inner rates, each kind of edge rate, first / interior / last
tiles of a run, odd and even surfaces, against the oracle, bit for bit."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu
RATES = [(0.95, 0.05), (1.0, 0.05), (0.95, 0.0), (0.5, 0.5), (0.3, 1.0), (0.0, 0.7), (1.0, 1.0), (2.0 ** -16, 0.999)]


@pytest.fixture(scope="module")
def eng():
    return engine()


@pytest.mark.parametrize("p,q", RATES)
@pytest.mark.parametrize("run,warps", [(1, 1), (2, 8), (4, 3)])
def test_work_queue(eng, p, q, run, warps):
    L = 512
    start = O.State.flat(L).run(3, 128, 128, 0.8, 0.3, seed=21)
    start.h00, start.t = -3, 6
    lat = eng.Lattice(L, p, q, seed=77, sample=5, run=run, warps_per_cta=warps)
    lat.set_slopes(start.packed(), h00=start.h00, t=start.t)
    start.run(3, 128, 128, p, q, 77, sample=5)
    r = lat.run(3).roughness()
    assert np.array_equal(lat.slopes(), start.packed())
    assert (r["S1"], r["S2"], r["h00"], r["t"]) == (*start.sums(), start.h00, start.t)
    lat.close()


def test_batch(eng):
    specs = [(256 << (k % 3), p, q, 13, k, 3 + k) for k, (p, q) in enumerate(RATES + [(1.0, 0.0)])]
    b = eng.Batch(specs, run=4, tile_y=128)
    b.run()
    s1, s2, h00 = b.sums()
    times = [int(t) for t in b.times()]
    for k, (L, p, q, seed, sample, n) in enumerate(specs):
        st = O.State.flat(L).run(n, 128, 128, p, q, seed, sample=sample)
        at = times.index(n)
        assert (int(s1[k, at]), int(s2[k, at]), int(h00[k])) == (*st.sums(), st.h00), (L, p, q)
    b.close()

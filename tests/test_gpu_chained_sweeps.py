"""Work-queue sweeps that follow one another in one launch, a chunk waiting only
for the rows of the sweep before that touch it: equal, bit for bit, to one launch
per sweep (kpz_run(1), which waits for nothing) and to the oracle. Lattices of
one row of tiles and of many, tall tiles, 2 x 2 cells, runs and block sizes, both
orders of taking and reporting chunks (few and many chunks a warp), and more
sweeps than rows."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu
RATES = [(1.0, 0.0), (0.95, 0.05), (0.5, 1.0)]


@pytest.fixture(scope="module")
def eng():
    return engine()


@pytest.mark.parametrize("L,knobs", [
    (128, dict(run=1)), (256, dict(run=1)), (256, dict(run=2, warps_per_cta=3)), (512, dict(run=1, warps_per_cta=1)),
    (256, dict(tile_y=256, run=1)), (1024, dict(tile_y=256, run=4, warps_per_cta=5)), (512, dict(cell=2)),
    (2048, dict(run=16)), (2048, dict(cell=2)), (4096, dict(tile_y=256)),
    (8192, dict()), (16384, dict()), (16384, dict(run=1))])
@pytest.mark.parametrize("p,q", RATES)
def test_against_one_launch_per_sweep(eng, L, knobs, p, q):
    many = eng.Lattice(L, p, q, seed=11, sample=2, **knobs)
    single = eng.Lattice(L, p, q, seed=11, sample=2, **knobs)
    for n in (2, 3, 41 if L < 8192 else 9):
        many.run(n)
        for _ in range(n):
            single.run(1)
        assert many.roughness() == single.roughness()
        assert np.array_equal(many.slopes(), single.slopes())
    many.close()
    single.close()


@pytest.mark.parametrize("L,knobs", [(128, dict(run=1)), (512, dict(run=1)), (512, dict(run=4, warps_per_cta=2))])
@pytest.mark.parametrize("p,q", RATES)
def test_against_oracle(eng, L, knobs, p, q):
    start = O.State.flat(L).run(2, 128, 128, 0.9, 0.4, seed=3)
    start.h00, start.t = 5, 11                      # odd parity, sweeps 11, 12, ...
    lat = eng.Lattice(L, p, q, seed=2 ** 40 + 7, sample=3, **knobs)
    lat.set_slopes(start.packed(), h00=start.h00, t=start.t)
    st = O.State(L, start.sx, start.sy)
    st.h00, st.t = start.h00, start.t
    for n in (2, 5):
        lat.run(n)
        st.run(n, 128, 128, p, q, 2 ** 40 + 7, sample=3)
        r = lat.roughness()
        assert np.array_equal(lat.slopes(), st.packed())
        assert (r["S1"], r["S2"], r["h00"], r["t"]) == (*st.sums(), st.h00, st.t)
    lat.close()

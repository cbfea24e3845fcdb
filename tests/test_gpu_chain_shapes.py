"""Chained work-queue sweeps (kpz_run calls of four or more sweeps with at least
1024 runs of tiles a sweep): every instantiation a caller reaches -- growth,
general rates with and without a 0 or 1, tall tiles, 2 x 2 cells -- equal, bit
for bit, to one launch per sweep and to the oracle, from an odd start parity and
a later sweep count, with more sweeps than rows of tiles and both orders of
taking and reporting chunks. The launches are counted, so a lattice that no
longer chains shows up here."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_5072_gb300._lib import launch_count
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu
GROWTH, INNER, EDGE = (1.0, 0.0), (0.95, 0.05), (0.5, 1.0)


@pytest.fixture(scope="module")
def eng():
    return engine()


def run_chained(lat, n):
    before = launch_count()
    lat.run(n)
    assert launch_count() - before == 2, "not chained"   # the sweeps, the sweep counter


@pytest.mark.parametrize("L,knobs,rates,counts", [
    (4096, dict(run=1), GROWTH, (4, 41)), (4096, dict(run=1, warps_per_cta=3), INNER, (4, 41)),
    (4096, dict(run=1, warps_per_cta=1), EDGE, (4, 41)),
    (8192, dict(tile_y=256), GROWTH, (5, 36)), (8192, dict(tile_y=256), INNER, (5, 36)),
    (8192, dict(tile_y=256, run=2, warps_per_cta=5), EDGE, (5, 36)),
    (16384, dict(tile_y=256, run=1), GROWTH, (4, 5)), (16384, dict(tile_y=256, run=1), INNER, (4, 5)),
    (4096, dict(cell=2, run=1), GROWTH, (4, 41)), (8192, dict(cell=2), GROWTH, (4, 9)),
    (16384, dict(), EDGE, (4, 9)), (16384, dict(run=1), INNER, (4, 9))])
def test_against_one_launch_per_sweep(eng, L, knobs, rates, counts):
    many = eng.Lattice(L, *rates, seed=2 ** 33 + 5, sample=2, **knobs)
    single = eng.Lattice(L, *rates, seed=2 ** 33 + 5, sample=2, **knobs)
    start = single.run(1).slopes()
    for lat in (many, single):
        lat.set_slopes(start, h00=7, t=12)          # odd parity, sweeps 12, 13, ...
    for n in counts:
        run_chained(many, n)
        for _ in range(n):
            single.run(1)
        assert many.roughness() == single.roughness()
        assert np.array_equal(many.slopes(), single.slopes())
    many.close()
    single.close()


@pytest.mark.parametrize("rates", [GROWTH, INNER, EDGE])
def test_against_oracle(eng, rates):
    L = 4096
    start = O.State.flat(L).run(1, 128, 128, 0.9, 0.4, seed=3)
    start.h00, start.t = 5, 11
    lat = eng.Lattice(L, *rates, seed=2 ** 40 + 7, sample=3, run=1)
    lat.set_slopes(start.packed(), h00=start.h00, t=start.t)
    run_chained(lat, 4)
    st = O.State(L, start.sx, start.sy)
    st.h00, st.t = start.h00, start.t
    st.run(4, 128, 128, *rates, 2 ** 40 + 7, sample=3)
    r = lat.roughness()
    assert np.array_equal(lat.slopes(), st.packed())
    assert (r["S1"], r["S2"], r["h00"], r["t"]) == (*st.sums(), st.h00, st.t)
    lat.close()

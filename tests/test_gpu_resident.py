"""Lattices swept by the resident kernels (no execution knobs given, up to 1024
tiles at a time): every layout -- one block, clusters of 4 and 16 blocks with
one and four tiles each, grids with one, two and seven tile warps per block --
against the oracle where it is quick and against the launch-per-sweep
kernels elsewhere, bit for bit; runs split over calls, odd start parity, tile sets."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu
RATES = [(1.0, 0.0), (0.95, 0.05), (0.5, 1.0), (0.0, 0.3)]


@pytest.fixture(scope="module")
def eng():
    return engine()


@pytest.mark.parametrize("L", [128, 256, 512, 1024])
@pytest.mark.parametrize("p,q", RATES)
def test_against_oracle(eng, L, p, q):
    start = O.State.flat(L).run(2, 128, 128, 0.9, 0.4, seed=3)
    start.h00, start.t = 5, 11                      # odd parity, sweeps 11, 12, ...
    lat = eng.Lattice(L, p, q, seed=2 ** 40 + 7, sample=3)
    lat.set_slopes(start.packed(), h00=start.h00, t=start.t)
    st = O.State(L, start.sx, start.sy)
    st.h00, st.t = start.h00, start.t
    for n in (1, 2, 3):
        lat.run(n)
        st.run(n, 128, 128, p, q, 2 ** 40 + 7, sample=3)
        r = lat.roughness()
        assert np.array_equal(lat.slopes(), st.packed())
        assert (r["S1"], r["S2"], r["h00"], r["t"]) == (*st.sums(), st.h00, st.t)
    lat.close()


@pytest.mark.parametrize("L", [256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("p,q", RATES)
@pytest.mark.parametrize("decomposition", [0, 1])
def test_against_launch_per_sweep(eng, L, p, q, decomposition):
    lat = eng.Lattice(L, p, q, seed=9, sample=1, decomposition=decomposition)
    ref = eng.Lattice(L, p, q, seed=9, sample=1, run=1, warps_per_cta=2, decomposition=decomposition)
    for n in (1, 4, 9):
        assert lat.run(n).roughness() == ref.run(n).roughness()
        assert np.array_equal(lat.slopes(), ref.slopes())
    lat.close()
    ref.close()


@pytest.mark.parametrize("decomposition", [0, 1])
def test_lattices_of_several_sizes_share_a_kernel(eng, decomposition):
    # A larger lattice still runs after smaller ones have been made, in any order.
    for p, q in ((1.0, 0.0), (0.95, 0.05)):
        lats = [eng.Lattice(L, p, q, seed=4, decomposition=decomposition) for L in (4096, 2048, 1024, 512, 256, 4096)]
        for lat in lats:
            lat.run(3)
        assert lats[0].roughness() == lats[-1].roughness()
        for lat in lats:
            lat.close()

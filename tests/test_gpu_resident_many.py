"""Many sweeps in one launch of the resident kernels against one launch per
sweep (execution knobs given), bit for bit: thousands of steps of each layout,
the tile that holds site (0,0) changing warps and diverging on its height in
most of them."""
import numpy as np
import pytest

from tests.gpu_util import engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    return engine()


def same_after(eng, L, p, q, decomposition, counts):
    lat = eng.Lattice(L, p, q, seed=21, sample=4, decomposition=decomposition)
    ref = eng.Lattice(L, p, q, seed=21, sample=4, decomposition=decomposition,
                      run=min(2, L // 128), warps_per_cta=2)
    for n in counts:
        assert lat.run(n).roughness() == ref.run(n).roughness()
        assert np.array_equal(lat.slopes(), ref.slopes())
    lat.close()
    ref.close()


# One and two tile warps a block with drawing warps, seven without; tile sets.
@pytest.mark.parametrize("L,p,q,decomposition", [
    (1024, 0.95, 0.05, 0), (2048, 1.0, 0.0, 0), (2048, 0.6, 0.3, 0), (4096, 1.0, 0.0, 0), (4096, 0.95, 0.05, 0),
    (2048, 0.95, 0.05, 1), (4096, 1.0, 0.0, 1), (4096, 0.6, 0.3, 1)])
def test_grid(eng, L, p, q, decomposition):
    same_after(eng, L, p, q, decomposition, (1000, 501))


# One block, a cluster of 4 and of 16 blocks with one and four units each; the
# drawing warps of a step run beside the tile warps of the step before.
@pytest.mark.parametrize("L,p,q,decomposition", [
    (128, 1.0, 0.0, 0), (256, 1.0, 0.0, 0), (512, 1.0, 0.0, 0), (1024, 1.0, 0.0, 0),
    (128, 0.95, 0.05, 0), (256, 0.6, 0.3, 0), (512, 0.95, 0.05, 0),
    (256, 1.0, 0.0, 1), (512, 0.95, 0.05, 1), (1024, 0.6, 0.3, 1), (1024, 1.0, 0.0, 1), (2048, 1.0, 0.0, 1)])
def test_cluster(eng, L, p, q, decomposition):
    same_after(eng, L, p, q, decomposition, (4000, 1501))


# The one shape in which tile sets run on seven tile warps a block that draw
# their own numbers; from an odd start parity and a later sweep count.
@pytest.mark.parametrize("p,q", [(1.0, 0.0), (0.95, 0.05), (0.5, 1.0)])
def test_tile_sets_without_drawing_warps(eng, p, q):
    L = 8192
    lat = eng.Lattice(L, p, q, seed=21, sample=4, decomposition=1)
    ref = eng.Lattice(L, p, q, seed=21, sample=4, decomposition=1, run=2, warps_per_cta=4)
    start = ref.run(1).slopes()
    for x in (lat, ref):
        x.set_slopes(start, h00=-5, t=9)
    for n in (1, 3, 40):
        assert lat.run(n).roughness() == ref.run(n).roughness()
        assert np.array_equal(lat.slopes(), ref.slopes())
    lat.close()
    ref.close()

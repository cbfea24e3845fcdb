"""Bounded device-side waits of kpz_run that run out: the launch ends by itself,
the next synchronising call answers KPZ_ETIMEOUT, the context is poisoned until
kpz_free, and the GPU and the buffer serve the next one. A counter in the
caller's buffer is set so that the awaited value never comes, and the bound to
50 ms (kpz_gridsync.cuh)."""
import time

import numpy as np
import pytest

from paper_1204_5072_gb300._lib import KPZ_ESTATE, KPZ_ETIMEOUT, KpzError
from tests.gpu_util import engine

pytestmark = pytest.mark.gpu

# Byte offsets from the block of small values behind the lattice.
QUEUE, ARRIVED, WAIT_MS = 48, 128, 128 + 12

KINDS = {
    # Grid barrier of the resident kernel: one arrival short of the first step.
    "resident": (dict(L=2048), ARRIVED),
    "resident tile sets, general rates": (dict(L=4096, p=0.95, q=0.05, decomposition=1), ARRIVED),
    # The first chunk of the first chained sweep is never taken from the queue.
    "chained": (dict(L=4096, run=1), QUEUE),
    "chained, general rates": (dict(L=8192, p=0.95, q=0.05), QUEUE),
    # Barrier of the random-sequential kernel.
    "random-sequential": (dict(L=256, decomposition=4), ARRIVED),
}
READS = {
    "roughness": lambda lat, path: lat.roughness(),
    "slopes": lambda lat, path: lat.slopes(),
    "heights": lambda lat, path: lat.heights(),
    "save": lambda lat, path: lat.save(path),
    "set_slopes": lambda lat, path: lat.set_slopes(np.zeros(lat.L * lat.L // 16, np.uint32)),
}


@pytest.fixture(scope="module")
def eng():
    return engine()


@pytest.mark.parametrize("kind,read", [(k, "roughness") for k in KINDS] + [("resident", r) for r in READS if r != "roughness"])
def test_wait_runs_out(eng, tmp_path, kind, read):
    import torch
    args, word = KINDS[kind]
    L = args["L"]
    buf = torch.empty(eng.Lattice.device_bytes(L), dtype=torch.uint8, device="cuda")
    small = (L * L // 8 + 255) // 256 * 256

    def poke(offset, value):
        buf[small + offset:small + offset + 4].view(torch.int32).fill_(value)

    lat = eng.Lattice(**args, seed=3, device_buffer=buf)
    want = lat.run(5).roughness()
    lat.reset()
    poke(WAIT_MS, 50)
    poke(word, 1 if word == QUEUE else -1)   # -1: the first arrival makes it 0
    t = time.perf_counter()
    lat.run(5)
    with pytest.raises(KpzError) as e:
        READS[read](lat, tmp_path / "ckpt")
    took = time.perf_counter() - t
    assert e.value.status == KPZ_ETIMEOUT and 0.05 <= took < 5.0
    for again in (lambda: lat.run(1), lat.roughness, lat.reset):
        with pytest.raises(KpzError) as e:
            again()
        assert e.value.status == KPZ_ESTATE
    lat.close()
    lat = eng.Lattice(**args, seed=3, device_buffer=buf)
    assert lat.run(5).roughness() == want
    lat.close()

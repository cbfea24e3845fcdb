"""kpz_init and kpz_free beside other work on the GPU: neither waits for more than
kpz.h says, and the caller's stream is not used when the memory is the caller's."""
import time

import pytest

from tests.gpu_util import engine

pytestmark = pytest.mark.gpu
L = 256


@pytest.fixture(scope="module")
def env():
    eng = engine()
    import torch
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    buf = torch.empty(eng.Lattice.device_bytes(L), dtype=torch.uint8, device="cuda")
    eng.Lattice(L, stream=a.cuda_stream, device_buffer=buf).close()   # first use of the kernels
    torch.cuda.synchronize()
    return eng, torch, a, b, buf


def busy(torch, stream):
    """About half a second of work on the stream."""
    with torch.cuda.stream(stream):
        torch.cuda._sleep(1_000_000_000)


def seconds(f):
    t = time.perf_counter()
    f()
    return time.perf_counter() - t


def test_free_leaves_the_callers_stream_alone(env):
    eng, torch, a, _, buf = env
    other = eng.Lattice(L)
    lat = eng.Lattice(L, stream=a.cuda_stream, device_buffer=buf)
    lat.run(2).roughness()
    busy(torch, a)
    took = seconds(lat.close)
    waited = seconds(torch.cuda.synchronize)
    other.close()
    assert took < 0.1 < waited


def test_stream_destroyed_before_free(env):
    eng, torch, _, _, buf = env
    import ctypes
    rt = torch.cuda.cudart()
    s = ctypes.c_void_p()
    assert int(rt.cudaStreamCreate(ctypes.addressof(s))) == 0
    lat = eng.Lattice(L, stream=s.value, device_buffer=buf)
    w2 = lat.run(2).roughness()["w2"]
    assert int(rt.cudaStreamDestroy(s.value)) == 0
    lat.close()
    again = eng.Lattice(L, device_buffer=buf)
    assert again.run(2).roughness()["w2"] == w2
    again.close()


def test_neither_waits_for_other_streams(env):
    # No other context is alive.
    eng, torch, a, b, buf = env
    lat = eng.Lattice(L, stream=a.cuda_stream, device_buffer=buf)
    lat.run(2).roughness()
    busy(torch, b)
    took = seconds(lat.close)
    took += seconds(lambda: eng.Lattice(L, stream=a.cuda_stream, device_buffer=buf).close())
    waited = seconds(torch.cuda.synchronize)
    assert took < 0.1 < waited

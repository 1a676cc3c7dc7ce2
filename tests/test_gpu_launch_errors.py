"""A launch that fails is reported by its own call and by no later one: a lattice
on the legacy default stream is stepped while another stream is being captured,
which CUDA refuses; after the capture every call works again."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, lbm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


def _runtime():
    with open("/proc/self/maps") as f:
        path = [line.split()[-1] for line in f if "libcudart" in line]
    if not path:
        pytest.skip("no shared CUDA runtime in this process")
    return ctypes.CDLL(path[0])


def _refused(step):
    rt = _runtime()
    stream = ctypes.c_void_p()   # one that synchronises with the legacy stream
    assert rt.cudaStreamCreate(ctypes.byref(stream)) == 0
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(stream, 0) == 0   # global mode
    try:
        with pytest.raises(Exception):
            step()
    finally:
        graph = ctypes.c_void_p()
        rt.cudaStreamEndCapture(stream, ctypes.byref(graph))
        rt.cudaGetLastError()
        assert rt.cudaStreamDestroy(stream) == 0


@pytest.mark.parametrize("algo", ["lptl", "nptl", "npol", "nsol", "aa"])
@pytest.mark.parametrize("dim", [2, 3])
def test_refused_step(dim, algo):
    lat = (lbm.Lattice(96, 40, 0.8, algo=algo) if dim == 2 else lbm.Lattice3(24, 12, 10, 0.8, algo=algo))
    lat.init()
    n = 96 * 40 if dim == 2 else 24 * 12 * 10
    _refused(lambda: lat.step(1))
    assert lat.mass() == pytest.approx(n, rel=1e-6)
    lat.init()
    lat.step(2).sync()
    assert lat.mass() == pytest.approx(n, rel=1e-6)


def test_refused_batch_step():
    b = lbm.Batch([lbm.make_params(60, 30, 0.8)] * 2, [np.zeros(1800, np.uint8)] * 2)
    _refused(lambda: b.step(1))
    b.step(2)
    b.sync()
    assert np.allclose(b.moments(1)[0], 1.0, rtol=1e-6)

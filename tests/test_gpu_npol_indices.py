"""NPOL's pulls by 32-bit indices over the lattice and the buffer grid against
the 64-bit ones (LBM_FLAG_WIDE_OFFSETS) and the two-lattice kernel, and its L2
prefetch, which changes no result. All of them read the same values and collide
them in the same order, so the states are equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, geometry as G, lbm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


def _state(nx, ny, steps, **kw):
    r = np.random.default_rng(nx + ny)
    mask = (r.random((ny, nx)) < 0.15).astype(np.uint8)
    mask[:, :2] = 0
    ux, uy = 0.02 + 1e-2 * r.standard_normal((2, ny, nx))
    lat = lbm.Lattice(nx, ny, 0.8, mask, force=(1e-5, -2e-5), **kw)
    h = lat.init(None, ux, uy).step(steps).populations("f64")
    lat.close()
    return h


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("layout", ["stream", "bundle", "collision"])
@pytest.mark.parametrize("size,tile", [((64, 8), (32, 8)), ((65, 9), (64, 4)), ((33, 17), (1, 1)), ((97, 34), (32, 4))])
def test_index_widths(size, tile, layout, storage):
    kw = dict(layout=layout, storage=storage)
    want = _state(*size, 7, algo="nptl", **kw)
    for flags in (0, lbm.LBM_FLAG_WIDE_OFFSETS):
        assert np.array_equal(_state(*size, 7, algo="npol", tile=tile, flags=flags, **kw), want), flags


def test_prefetch():
    nx, ny = 2048, 2560   # FP32 populations beyond the L2 cache
    mask = G.porous_discs(nx, ny, seed=5)
    got = []
    for flags in (0, lbm.LBM_FLAG_NO_PREFETCH):
        lat = lbm.Lattice(nx, ny, 0.8, mask, force=(1e-5, 0.0), layout="bundle", algo="npol", tile=(64, 4),
                          storage="f32", flags=flags)
        assert (lat.info()["prefetch_distance"] > 0) == (flags == 0)
        got.append(lat.init(None, np.full(nx * ny, 0.02), None).step(5).populations("f32"))
        lat.close()
    assert np.array_equal(*got)

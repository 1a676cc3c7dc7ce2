"""16-bit node pairs pulled by 32-bit words: bit-identical to one node per
thread on narrow lattices, on warps with and without bounced links, with solid
partners on either side, and over every edge kind."""
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


@pytest.mark.parametrize("storage", ["f16s", "bf16s"])
@pytest.mark.parametrize("rounding", ["rne", "sr"])
@pytest.mark.parametrize("nx,ny", [(2, 3), (4, 4), (64, 9), (66, 17), (256, 20)])
def test_words(nx, ny, rounding, storage):
    r = np.random.default_rng(nx)
    ux, uy = 2e-2 * r.standard_normal((2, ny, nx))
    for solid in (0.0, 0.02, 0.5):
        mask = (r.random((ny, nx)) < solid).astype(np.uint8)
        for bc in ((lbm.PERIODIC,) * 4, (lbm.WALL, lbm.OUTFLOW_ZG, lbm.FREESLIP, lbm.WALL)):
            for algo in ("lptl", "nptl"):
                got = []
                for flags in (0, lbm.LBM_FLAG_NO_PAIRS):
                    lat = lbm.Lattice(nx, ny, 0.8, mask, force=(1e-4, -1e-4), bc=bc, layout="bundle", algo=algo,
                                      storage=storage, rounding=rounding, seed=3, flags=flags).init(None, ux, uy)
                    lat.step(5, moments=True)
                    got.append([lat.populations()] + list(lat.moments()))
                for a, b in zip(*got):
                    assert np.array_equal(a, b), (solid, bc, algo)

"""Small lattices, whose tiles are cut into smaller blocks: LPTL, NPTL and the
AA pattern equal NPOL (whose tiles stay whole) bit for bit around the sizes
where the cut begins, with even and odd tile heights and rows left over."""
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


# 4 blocks per SM on 152 SMs: cut below 608 blocks; 32 x 8 tiles of 512 x 304
# nodes are 608 blocks, of 512 x 303 too (ragged), of 512 x 296 are 592
@pytest.mark.parametrize("nx,ny,tile", [(512, 304, (32, 8)), (512, 303, (32, 8)), (512, 296, (32, 8)),
                                        (256, 64, (32, 8)), (100, 37, (64, 4)), (96, 50, (32, 5)), (33, 9, (128, 1)),
                                        (40, 21, (8, 4))])
def test_cut_blocks(nx, ny, tile):
    r = np.random.default_rng(ny)
    mask = (r.random((ny, nx)) < 0.1).astype(np.uint8)
    ux, uy = 1e-2 * r.standard_normal((2, ny, nx))
    kw = dict(force=(1e-5, 0.0), bc=(lbm.PERIODIC, lbm.PERIODIC, lbm.FREESLIP, lbm.WALL), layout="bundle")
    for storage in ("f32", "f64"):
        ref = lbm.Lattice(nx, ny, 0.8, mask, algo="npol", tile=tile, storage=storage, **kw).init(None, ux, uy)
        ref.step(6, moments=True)
        want, mom = ref.populations(), ref.moments()
        for algo in ("lptl", "nptl", "aa"):
            lat = lbm.Lattice(nx, ny, 0.8, mask, algo=algo, tile=tile, storage=storage, **kw).init(None, ux, uy)
            lat.step(4).step(2, moments=True)
            assert np.array_equal(lat.populations(), want), (algo, storage)
            for a, b in zip(lat.moments(), mom):
                assert np.array_equal(a, b), (algo, storage)

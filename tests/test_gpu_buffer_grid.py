"""Addressing of the one-lattice algorithms' buffer grid: NPOL and NSOL equal
NPTL bit for bit where a tile spans a whole axis, ends one node short of the
edge, is one node wide, or is larger than the lattice."""
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


EDGES = {"periodic": (lbm.PERIODIC,) * 4,
         "channel": (lbm.INLET_ZOUHE, lbm.OUTFLOW_ZG, lbm.FREESLIP, lbm.WALL),
         "box": (lbm.WALL, lbm.WALL, lbm.FREESLIP, lbm.FREESLIP)}


@pytest.mark.parametrize("edges", EDGES)
@pytest.mark.parametrize("size,tile", [((64, 8), (32, 8)), ((65, 9), (64, 4)), ((33, 17), (1, 1)), ((40, 6), (64, 8)),
                                       ((31, 30), (31, 5)), ((96, 33), (32, 4)), ((7, 5), (4, 2))])
def test_2d(size, tile, edges):
    nx, ny = size
    r = np.random.default_rng(nx)
    mask = (r.random((ny, nx)) < 0.15).astype(np.uint8)
    mask[:, :2] = 0
    ux, uy = 0.02 + 1e-2 * r.standard_normal((2, ny, nx))
    kw = dict(force=(1e-5, -2e-5), u_in=(0.03, 0.0), bc=EDGES[edges], storage="f32")
    for layout in ("stream", "bundle", "collision"):
        want = lbm.Lattice(nx, ny, 0.8, mask, layout=layout, **kw).init(None, ux, uy).step(7).populations("f32")
        for algo in ("npol", "nsol"):
            got = lbm.Lattice(nx, ny, 0.8, mask, layout=layout, algo=algo, tile=tile, **kw).init(None, ux, uy)
            assert np.array_equal(got.step(7).populations("f32"), want), (layout, algo)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size,tile", [((8, 8, 8), (8, 8, 8)), ((9, 8, 7), (4, 3, 2)), ((5, 6, 7), (8, 2, 1)),
                                       ((3, 1, 4), (1, 1, 1)), ((12, 5, 9), (128, 1, 1)), ((17, 9, 9), (16, 8, 4))])
def test_3d(size, tile, walls):
    nx, ny, nz = size
    r = np.random.default_rng(nx)
    mask = (r.random((nz, ny, nx)) < 0.1).astype(np.uint8)
    u = 1e-2 * r.standard_normal((3, nz, ny, nx))
    kw = dict(force=(1e-5, 0.0, -2e-5), bc=(lbm.PERIODIC,) + ((lbm.WALL,) if walls else (lbm.PERIODIC,)) * 2, storage="f32")
    for layout in ("stream", "bundle", "collision"):
        want = lbm.Lattice3(nx, ny, nz, 0.8, mask, layout=layout, **kw).init(None, *u).step(5).populations("f32")
        for algo in ("npol", "nsol"):
            for flags in (0, lbm.LBM_FLAG_WIDE_OFFSETS):
                got = lbm.Lattice3(nx, ny, nz, 0.8, mask, layout=layout, algo=algo, tile=tile, flags=flags, **kw)
                assert np.array_equal(got.init(None, *u).step(5).populations("f32"), want), (layout, algo, flags)

"""The interior pulls by indices, by pointers and of warps without a bounced link,
and the launches on both sides of the size from which updates are not chained.
All of them read the same values and collide them in the same order, so every
state equals the buffer-grid kernel's, which has pulls of its own, bit for bit."""
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


def _flow(nx, ny, solid):
    r = np.random.default_rng(nx + ny)
    mask = np.zeros((ny, nx), np.uint8)
    if solid:
        mask[r.integers(0, ny, solid), r.integers(0, nx, solid)] = 1
    ux, uy = 0.02 + 1e-2 * r.standard_normal((2, ny, nx))
    return mask, ux, uy


@pytest.mark.parametrize("layout", ["stream", "bundle", "collision"])
@pytest.mark.parametrize("ny", [2048, 2049])   # 4M nodes: the last chained size; one row more
def test_both_sides_of_the_chained_sizes(ny, layout):
    nx = 2048
    mask, ux, uy = _flow(nx, ny, 20000)
    want = None
    for algo, tile in (("npol", (64, 4)), ("nptl", (32, 4)), ("lptl", (0, 0)), ("aa", (64, 2))):
        lat = lbm.Lattice(nx, ny, 0.8, mask, force=(1e-5, -2e-5), layout=layout, algo=algo, tile=tile, storage="f32")
        got = lat.init(None, ux, uy).step(4).populations("f32")
        lat.close()
        want = got if want is None else want
        assert np.array_equal(got, want), algo


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("layout", ["stream", "bundle", "collision"])
@pytest.mark.parametrize("algo", ["lptl", "nptl"])
def test_batches(algo, layout, storage):
    sizes = [(130, 70, 0), (130, 70, 5), (64, 33, 300), (1, 40, 0), (300, 2, 3)]
    kw = dict(force=(1e-5, 0.0), layout=layout, storage=storage)
    tile = (0, 0) if algo == "lptl" else (32, 4)
    flows = [_flow(*s) for s in sizes]
    batch = lbm.Batch([lbm.make_params(nx, ny, 0.8, algo=algo, tile=tile, **kw) for nx, ny, _ in sizes],
                      [f[0] for f in flows])
    for c, f in enumerate(flows):
        batch.init(c, None, f[1], f[2])
    batch.step(7).sync()
    for c, ((nx, ny, _), f) in enumerate(zip(sizes, flows)):
        lat = lbm.Lattice(nx, ny, 0.8, f[0], algo="npol", tile=(32, 4), **kw).init(None, f[1], f[2])
        assert np.array_equal(batch.populations(c), lat.step(7).populations()), c
        lat.close()
    batch.close()

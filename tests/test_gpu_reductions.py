"""Second pass of the mass and force reductions (a tree over the block
partials that also hands the error word to the host): against the FP64 oracle
where fewer, exactly and more than one node per first-pass thread contribute,
and a non-finite density seen by an update is reported by either call."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, geometry as G, lbm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


# 1024 blocks of 256 threads: below one node per thread, one, and several
@pytest.mark.parametrize("nx,ny", [(7, 5), (512, 512), (1031, 517)])
def test_mass_and_force_2d(nx, ny):
    r = np.random.default_rng(nx)
    mask = G.disc(nx, ny, nx / 3, ny / 2, max(1.0, ny / 6))
    rho = 1 + 1e-2 * r.standard_normal((ny, nx))
    ux, uy = 1e-2 * r.standard_normal((2, ny, nx))
    ref = O.Lattice(O.Case(nx, ny, 0.8, fx=1e-6), mask, rho=rho, ux=ux, uy=uy)
    with_f64 = lbm.Lattice(nx, ny, 0.8, mask, force=(1e-6, 0.0), storage="f64").init(rho, ux, uy)
    # sums of n terms in another order: n ulp of the sum of magnitudes at the very most, sqrt(n) in the mean
    n = nx * ny
    assert abs(with_f64.mass() - ref.mass()) <= 4e-16 * np.sqrt(n) * n + 1e-12
    want = ref.force(mask)
    links = 8 * n ** 0.5 * 9
    assert np.abs(with_f64.force(torch.from_numpy(mask.reshape(-1)).cuda()) - want).max() <= 1e-15 * links + 1e-13
    assert with_f64.mass() == with_f64.mass()   # fixed order: the same bits


def test_mass_and_force_3d():
    n = (70, 41, 33)
    r = np.random.default_rng(3)
    mask = G.ball(*n, 20, 20, 16, 7.5)
    ux, uy, uz = 1e-2 * r.standard_normal((3,) + n[::-1])
    ref = O.Lattice3(O.Case3(*n, 0.8, 0.0, 0.0, 0.0), mask, ux=ux, uy=uy, uz=uz)
    lat = lbm.Lattice3(*n, 0.8, mask, storage="f64").init(None, ux, uy, uz)
    assert abs(lat.mass() - ref.mass()) <= 4e-16 * mask.size ** 1.5
    assert np.abs(lat.force() - ref.force(mask)).max() <= 1e-11   # ~10^4 links of ~0.1


@pytest.mark.parametrize("call", ["mass", "force"])
@pytest.mark.parametrize("dim", [2, 3])
def test_divergence_is_reported(call, dim):
    lat = lbm.Lattice(64, 48, 0.8) if dim == 2 else lbm.Lattice3(24, 20, 16, 0.8)
    h = lat.populations()
    h[3, 100] = np.nan
    lat.write_populations(h)
    lat.step(1)
    with pytest.raises(lbm.LbmError) as e:
        getattr(lat, call)()
    assert e.value.status == lbm.LBM_EDIVERGED
    lat.sync()   # the flag was cleared

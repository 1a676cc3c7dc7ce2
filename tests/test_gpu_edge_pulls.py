"""Pulls of nodes on the domain edge: every pair of edge kinds, in every layout,
on lattices whose warps mix edge and inner nodes or hold edge nodes only,
against the FP64 oracle."""
import itertools

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, lbm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


WEST_EAST = [(lbm.PERIODIC, lbm.PERIODIC)] + list(itertools.product(
    (lbm.WALL, lbm.INLET_ZOUHE, lbm.INLET_EQ, lbm.OUTFLOW_ZG, lbm.INLET_EQ_NEUMANN),
    (lbm.WALL, lbm.OUTFLOW_ZG, lbm.OUTLET_PRESSURE)))
SOUTH_NORTH = [(lbm.PERIODIC, lbm.PERIODIC)] + list(itertools.product((lbm.WALL, lbm.FREESLIP), repeat=2))


@pytest.mark.parametrize("size", [(2, 1), (5, 3), (70, 6), (33, 40)])
@pytest.mark.parametrize("sn", SOUTH_NORTH)
def test_every_pair_of_edges(size, sn):
    nx, ny = size
    r = np.random.default_rng(nx)
    mask = (r.random((ny, nx)) < 0.1).astype(np.uint8)
    mask[:, :2] = 0
    rho = 1 + 1e-2 * r.standard_normal((ny, nx))
    ux, uy = 2e-2 * r.standard_normal((2, ny, nx))
    for we in WEST_EAST:
        bc = we + sn
        ref = O.Lattice(O.Case(nx, ny, 0.8, fx=1e-4, fy=-2e-4, ux_in=0.02, uy_in=0.01, bc_w=bc[0], bc_e=bc[1],
                               bc_s=bc[2], bc_n=bc[3], rho_out=1.01), mask, rho=rho, ux=ux, uy=uy).run(6)
        want = ref.h.reshape(9, -1)
        for layout, algo in itertools.product(("stream", "bundle", "collision"), ("lptl", "nptl")):
            lat = lbm.Lattice(nx, ny, 0.8, mask, force=(1e-4, -2e-4), u_in=(0.02, 0.01), bc=bc, rho_out=1.01,
                              layout=layout, algo=algo, storage="f64").init(rho, ux, uy)
            got = lat.step(6).populations()
            # a few roundings of values of ~1e-2 in each of six updates
            assert np.abs(got - want).max() <= 1e-15, (bc, layout, algo)

"""Batched ensembles: one persistent launch per update over all cases must
give, for every case, exactly the bits of a single-lattice run of that case
(same arithmetic, only the scheduling differs)."""
import numpy as np
import pytest

from tests.gpu_helpers import COMBOS

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, geometry as G, lbm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


def _cases(n, seed=9):
    return G.batch_channels(ncases=n, seed=seed, wmin=20, wmax=140, hmin=9, hmax=70)


def _params(w, storage="f32", rounding="rne", **kw):
    return lbm.make_params(w.nx, w.ny, w.tau, u_in=(w.ux_in, 0.0), bc=(w.bc_w, w.bc_e, w.bc_s, w.bc_n),
                           storage=storage, rounding=rounding, seed=77, **kw)


@pytest.mark.parametrize("storage,rounding", [("f32", "rne"), ("f16s", "sr"), ("f64", "rne")])
def test_batch_equals_single_runs_for_every_combination(storage, rounding):
    ws = _cases(len(COMBOS) + 3)
    params = []
    for k, w in enumerate(ws):
        layout, algo = COMBOS[k % len(COMBOS)]
        tile = (0, 0) if algo == "lptl" else [(32, 8), (64, 4), (16, 16), (32, 2)][k % 4]
        params.append(_params(w, storage, rounding, layout=layout, algo=algo, tile=tile))
    b = lbm.Batch(params, [w.mask for w in ws], plan=False)
    for c, w in enumerate(ws):
        b.init(c, None, w.ux0, w.uy0)
    T = 137                    # one 100-update graph plus a remainder
    b.step(T, moments=True).sync()
    for c, w in enumerate(ws):
        single = lbm.Lattice(w.nx, w.ny, w.tau, w.mask, u_in=(w.ux_in, 0.0),
                             bc=(w.bc_w, w.bc_e, w.bc_s, w.bc_n), layout="stream", algo="nptl",
                             storage=storage, rounding=rounding, seed=77)
        single.init(None, w.ux0, w.uy0)
        single.step(T, moments=True).sync()
        assert np.array_equal(b.populations(c), single.populations()), c
        for x, y in zip(b.moments(c), single.moments()):
            assert np.array_equal(x, y), c
        single.close()
    info = b.info()
    assert info["tiles"] > len(ws) and info["grid"] >= 1
    b.close()


def test_autotuned_batch_equals_single_runs():
    ws = _cases(10, seed=13)
    probe = lbm.make_params(512, 256, 0.8, storage="f32")
    mask = G.porous_discs(512, 256, seed=3, rmin=8, rmax=16)
    nbytes = lbm.lbm_tune_workspace_bytes(probe)
    wsp = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    tuning = lbm.lbm_tune(probe, mask, wsp, nbytes, lbm.current_stream())
    assert tuning.valid == 1
    ns = np.array([[tuning.ns_per_cell[l][a] for a in range(4)] for l in range(3)])
    assert (ns > 0).all() and np.isfinite(ns).all()
    params = [_params(w, layout=lbm.LBM_AUTO, algo=lbm.LBM_AUTO) for w in ws]
    b = lbm.Batch(params, [w.mask for w in ws], tuning=tuning)
    for c, w in enumerate(ws):
        b.init(c, None, w.ux0, w.uy0)
    b.step(60).sync()
    for c, w in enumerate(ws):
        single = lbm.Lattice(w.nx, w.ny, w.tau, w.mask, u_in=(w.ux_in, 0.0),
                             bc=(w.bc_w, w.bc_e, w.bc_s, w.bc_n), storage="f32")
        single.init(None, w.ux0, w.uy0)
        single.step(60).sync()
        assert np.array_equal(b.populations(c), single.populations()), c
        single.close()
    with pytest.raises(lbm.LbmError):
        b.init(0)
    b.close()


def test_each_case_declines_the_prefetch_for_itself():
    """Device records of batches beyond the L2 cache: LBM_FLAG_NO_PREFETCH of a case changes its own
    records (one per parity and moments flag) and no other's, whichever case sets it."""
    nx, ny, n = 2048, 1024, 3
    masks = [np.zeros(nx * ny, np.uint8)] * n
    base = [lbm.make_params(nx, ny, 0.8, layout="bundle", algo="lptl", storage="f32") for _ in range(n)]
    nbytes = lbm.lbm_batch_workspace_bytes(base)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

    def records(declining):
        ws[: 1 << 16].zero_()
        ps = [lbm.make_params(nx, ny, 0.8, layout="bundle", algo="lptl", storage="f32",
                              flags=lbm.LBM_FLAG_NO_PREFETCH if c in declining else 0) for c in range(n)]
        h = lbm.lbm_batch_create(ps, masks, ws, nbytes, torch.cuda.current_stream().cuda_stream)[0]
        torch.cuda.synchronize()
        out = ws[: 1 << 14].cpu().numpy().view(np.int32).copy()   # 12 records and the first work items
        lbm.lbm_batch_destroy(h)
        return out

    none = records(())
    where = [np.nonzero(records((c,)) != none)[0] for c in range(n)]
    assert all(len(w) == 4 for w in where)
    assert len(set(np.concatenate(where))) == 4 * n
    assert np.array_equal(np.sort(np.concatenate(where[:2])), np.nonzero(records((0, 1)) != none)[0])

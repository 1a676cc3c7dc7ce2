"""The fixed operation order of the 16-bit collision, D2Q9 and D3Q19: every
rounded FP32 operation is repeated here in numpy (fma included) and the stored
16-bit populations have to agree to the last bit, one node and packed pairs, with
and without a force, also at relaxation times whose product with the force
exceeds the FP32 range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, lbm  # noqa: E402

f32 = np.float32
D2 = [(i % 3 - 1, i // 3 - 1) for i in range(9)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


def _fma(a, b, c):
    """a b + c of FP32 values, rounded once: the product is exact in FP64, the
    sum is rounded to odd there, which makes the second rounding exact."""
    p = np.asarray(a, np.float64) * np.asarray(b, np.float64)
    c = np.asarray(c, np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    odd = np.asarray(s).view(np.uint64) & np.uint64(1)
    s = np.where((err != 0) & (odd == 0), np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return s.astype(f32)


def _relax(g, cu, sg3, base, m3uF, w, wl, kw, cF, omega, force):
    P = base if cu is None else _fma(cu, _fma(f32(4.5), cu, sg3), base)
    t = _fma(-wl, P, _fma(-w, P, g))
    o = _fma(-omega, t, g)
    if force:
        o = _fma(kw, m3uF if cu is None else _fma(cF, _fma(f32(9), cu, sg3), m3uF), o)
    return o


def _weights(ws, omega64):
    w = [f32(v) for v in ws]
    return w, [f32(v - float(r)) for v, r in zip(ws, w)], [f32((1 - 0.5 * omega64) * v) for v in ws]


def _collide2(g, omega64, F):
    w, wl, kw = _weights([1 / 36, 1 / 9, 4 / 9], omega64)
    kw = [f32((1 - 0.5 * omega64) / 36), f32((1 - 0.5 * omega64) / 9), f32(4 * (1 - 0.5 * omega64) / 9)]
    fx, fy = f32(F[0]), f32(F[1])
    drho = ((g[0] + g[3] + g[6]) + (g[1] + g[4] + g[7])) + (g[2] + g[5] + g[8])
    ux = ((g[2] + g[5] + g[8]) - (g[0] + g[3] + g[6])) + f32(0.5 * F[0])
    uy = ((g[6] + g[7] + g[8]) - (g[0] + g[1] + g[2])) + f32(0.5 * F[1])
    base = _fma(f32(-1.5), _fma(ux, ux, uy * uy), drho)
    m3uF = f32(-3) * _fma(ux, fx, uy * fy)
    pair = {0: (ux + uy, f32(F[0] + F[1])), 1: (uy, fy), 2: (ux - uy, f32(F[0] - F[1])), 3: (ux, fx)}
    pair.update({8: pair[0], 7: pair[1], 6: pair[2], 5: pair[3]})
    out = []
    for i in range(9):
        c, cF = (None, None) if i == 4 else pair[i]
        s = 2 if i == 4 else (1 if i & 1 else 0)
        sg3 = f32(3) if i in (2, 5, 7, 8) else f32(-3)
        out.append(_relax(g[i], c, sg3, base, m3uF, w[s], wl[s], kw[s], cF, f32(omega64), any(F)))
    return np.stack(out)


def _collide3(g, omega64, F, C):
    w, wl, _ = _weights([1 / 3, 1 / 18, 1 / 36], omega64)
    kw = [f32((1 - 0.5 * omega64) / d) for d in (3, 18, 36)]
    drho = g[0]
    for i in range(1, 19):
        drho = drho + g[i]
    u = [None] * 3
    for i in range(19):
        for a in range(3):
            if C[i][a]:
                t = g[i] if C[i][a] > 0 else -g[i]
                u[a] = t if u[a] is None else u[a] + t
    u = [v + f32(0.5 * f) for v, f in zip(u, F)]
    base = _fma(f32(-1.5), _fma(u[0], u[0], _fma(u[1], u[1], u[2] * u[2])), drho)
    m3uF = f32(-3) * _fma(u[0], f32(F[0]), _fma(u[1], f32(F[1]), u[2] * f32(F[2])))
    out = []
    for i in range(19):
        cu = None
        for a in range(3):
            if C[i][a]:
                t = u[a] if C[i][a] > 0 else -u[a]
                cu = t if cu is None else cu + t
        s = int(sum(v * v for v in C[i]))
        cF = f32(sum(int(v) * f for v, f in zip(C[i], F)))
        out.append(_relax(g[i], cu, f32(3), base, m3uF, w[s], wl[s], kw[s], cF, f32(omega64), any(F)))
    return np.stack(out)


def _stored(x, storage):
    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.float16 if storage == "f16s" else torch.bfloat16) \
        .float().numpy()


# tau, F: without a force, with one, and with tau F beyond FP32 (4e38)
FLOWS = [(0.8, 0.0), (0.56, 3e-4), (1e3, 1e-3), (1e41, 1e-3)]


@pytest.mark.parametrize("storage", ["f16s", "bf16s"])
@pytest.mark.parametrize("tau,f", FLOWS)
@pytest.mark.parametrize("kw", [{"layout": "bundle", "algo": "nptl"}, {"layout": "bundle", "algo": "lptl"},
                                {"layout": "stream", "algo": "nptl"}, {"layout": "bundle", "algo": "npol"}],
                         ids=["pairs", "linear pairs", "one node", "npol"])
def test_d2q9(storage, tau, f, kw):
    nx, ny = 70, 19
    F = (f, -0.4 * f)
    h = _stored((2e-2 * np.random.default_rng(5).standard_normal((9, ny, nx))).astype(f32), storage)
    lat = lbm.Lattice(nx, ny, tau, force=F, bc=(lbm.PERIODIC,) * 4, storage=storage, **kw)
    lat.write_populations(h.reshape(9, -1))
    for _ in range(3):
        g = np.stack([np.roll(h[i], (D2[i][1], D2[i][0]), axis=(0, 1)) for i in range(9)])
        h = _stored(_collide2(g, 1.0 / tau, F), storage)
        lat.step(1).sync()
        assert np.array_equal(lat.populations("f32").reshape(h.shape), h)
    assert np.isfinite(h).all()


@pytest.mark.parametrize("storage", ["f16s", "bf16s"])
@pytest.mark.parametrize("tau,f", FLOWS)
@pytest.mark.parametrize("kw", [{"layout": "bundle", "algo": "nptl"}, {"layout": "collision", "algo": "lptl"}],
                         ids=["pairs", "one node"])
def test_d3q19(storage, tau, f, kw):
    import oracle
    C = [tuple(int(v) for v in c) for c in oracle.directions3()[0]]
    nx, ny, nz = 34, 9, 7
    F = (f, -0.4 * f, 0.3 * f)
    h = _stored((2e-2 * np.random.default_rng(6).standard_normal((19, nz, ny, nx))).astype(f32), storage)
    box = lbm.Lattice3(nx, ny, nz, tau, force=F, storage=storage, **kw)
    box.write_populations(h.reshape(19, -1))
    for _ in range(3):
        g = np.stack([np.roll(h[i], C[i][::-1], axis=(0, 1, 2)) for i in range(19)])
        h = _stored(_collide3(g, 1.0 / tau, F, C), storage)
        box.step(1).sync()
        assert np.array_equal(box.populations("f32").reshape(h.shape), h)
    assert np.isfinite(h).all()

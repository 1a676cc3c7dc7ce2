"""State and moments between device and host: around the sizes from which they
go through the thread's page-locked slots (1 MB of populations, 8 MB of one
moments field), page-locked and unaligned buffers, an array that numpy holds
read-only (read-only pages: test_gpu_shared_host.py), every layout, slot order
and storage type."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, lbm  # noqa: E402

DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


def _rounded(h, storage):
    t = torch.from_numpy(h)
    return (t if storage == "f64" else t.float().to(DTYPE[storage])).double().numpy()


# 9 x 14,563 doubles are just below 1 MiB, 14,564 just above; the last is far above
@pytest.mark.parametrize("nx,ny", [(3, 5), (14563, 1), (14564, 1), (331, 257)])
@pytest.mark.parametrize("layout", ["stream", "bundle", "collision"])
def test_state_2d(nx, ny, layout):
    r = np.random.default_rng(nx)
    N = nx * ny
    mask = (r.random(N) < 0.2).astype(np.uint8)
    h = 1e-2 * r.standard_normal((9, N))
    for storage in DTYPE:
        for algo in ("nptl", "npol", "nsol", "aa"):
            lat = lbm.Lattice(nx, ny, 0.8, mask.reshape(ny, nx), layout=layout, algo=algo, storage=storage)
            for src in (h, h.astype(np.float32)):
                lat.write_populations(src)
                got = lat.populations("f64")
                solid = (got == 0).all(axis=0)   # given solids and enclosed nodes
                assert solid[mask > 0].all()
                want = np.where(solid, 0.0, _rounded(src.astype(np.float64), storage))
                assert np.array_equal(got, want)
                assert np.array_equal(lat.populations("f32"), want.astype(np.float32))
            raw = lat.workspace[: 9 * N * DTYPE[storage].itemsize].view(DTYPE[storage]).double().cpu().numpy()
            for n, i in zip(r.integers(0, N, 50), r.integers(0, 9, 50)):
                slot = 8 - i if algo in ("nsol", "aa") else i
                assert raw[lbm.lbm_layout_index(layout, N, int(n), int(slot))] == want[i, n]


@pytest.mark.parametrize("shape", [(5, 4, 3), (47, 31, 29)])
def test_state_3d(shape):
    nx, ny, nz = shape
    N = nx * ny * nz
    r = np.random.default_rng(nx)
    h = 1e-2 * r.standard_normal((19, N))
    for storage in DTYPE:
        for layout in ("stream", "bundle", "collision"):
            for algo in ("nptl", "npol", "nsol"):
                lat = lbm.Lattice3(nx, ny, nz, 0.8, layout=layout, algo=algo, storage=storage)
                lat.write_populations(h)
                want = _rounded(h, storage)
                assert np.array_equal(lat.populations("f64"), want)
                assert np.array_equal(lat.populations("f32"), want.astype(np.float32))
                raw = lat.workspace[: 19 * N * DTYPE[storage].itemsize].view(DTYPE[storage]).double().cpu().numpy()
                for n, i in zip(r.integers(0, N, 50), r.integers(0, 19, 50)):
                    slot = 18 - i if algo == "nsol" else i
                    assert raw[lbm.lbm3_layout_index(layout, N, int(n), int(slot))] == want[i, n]


def test_unaligned_page_locked_and_read_only_buffers():
    nx, ny = 331, 257
    N = nx * ny
    lat = lbm.Lattice(nx, ny, 0.8, storage="f32")
    h = (1e-2 * np.random.default_rng(1).standard_normal((9, N))).astype(np.float32).astype(np.float64)
    ro = h.copy()
    ro.setflags(write=False)
    lat.write_populations(ro)
    big = np.empty(9 * N + 64)
    for shift in (1, 7):
        out = big[shift: shift + 9 * N]
        big[:] = -1.0
        assert lbm.load().lbm_read_populations(lat.h, out.ctypes.data, 0) == 0
        assert np.array_equal(out.reshape(9, N), h)
        assert (big[:shift] == -1.0).all() and (big[shift + 9 * N:] == -1.0).all()
    pinned = torch.empty(9 * N, dtype=torch.float64, pin_memory=True).numpy()
    assert lbm.load().lbm_read_populations(lat.h, pinned.ctypes.data, 0) == 0
    assert np.array_equal(pinned.reshape(9, N), h)
    assert lbm.load().lbm_write_populations(lat.h, pinned.ctypes.data, 0) == 0
    assert np.array_equal(lat.populations(), h)


@pytest.mark.parametrize("N", [1 << 18, (1 << 18) + 1, (1 << 20) - 1, 1 << 20])
def test_moments_around_the_thresholds(N):
    r = np.random.default_rng(N)
    ux, uy = 1e-2 * r.standard_normal((2, N))
    lat = lbm.Lattice(N, 1, 0.8, storage="f32").init(1 + ux, ux, uy)
    dev = [torch.empty(N, dtype=torch.float32, device="cuda") for _ in range(3)]
    lbm.lbm_moments_device(lat.h, *dev)
    want = [d.double().cpu().numpy() for d in dev]
    for a, b in zip(lat.moments(), want):
        assert np.array_equal(a, b)
    only = np.empty(N)
    assert lbm.load().lbm_read_moments(lat.h, None, None, only.ctypes.data) == 0
    assert np.array_equal(only, want[2])
    box = lbm.Lattice3(N, 1, 1, 0.8, storage="f32").init(1 + ux, ux, uy, -ux)
    got = box.moments()
    for a, b in zip(got, (1 + ux, ux, uy, -ux)):
        assert np.abs(a - b).max() <= 2.0 ** -20   # FP32 sums of values below 1


@pytest.mark.parametrize("N", [1, 1000, 32768, 32769, 43690, 43691])   # scratch: 2^20 bytes of three or four fields
def test_fp64_moments_around_the_scratch_buffer(N):
    r = np.random.default_rng(N)
    ux, uy = 1e-2 * r.standard_normal((2, N))
    lat = lbm.Lattice(N, 1, 0.8, storage="f64").init(1 + ux, ux, uy)
    box = lbm.Lattice3(N, 1, 1, 0.8, storage="f64").init(1 + ux, ux, uy, -ux)
    for got, want in ((lat.moments(), (1 + ux, ux, uy)), (box.moments(), (1 + ux, ux, uy, -ux))):
        for a, b in zip(got, want):
            assert np.abs(a.reshape(-1) - b).max() <= 2.0 ** -49   # FP64 sums of values below 2
    only = np.empty(N)
    assert lbm.load().lbm_read_moments(lat.h, None, only.ctypes.data, None) == 0
    assert np.array_equal(only, lat.moments()[1].reshape(-1))


@pytest.mark.parametrize("N", [8192, 8193])   # fields of 64 KB and one value more
@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_moments_into_locked_memory_around_64_kb(N, storage):
    r = np.random.default_rng(N)
    ux, uy = 1e-2 * r.standard_normal((2, N))
    lat = lbm.Lattice(N, 1, 0.8, storage=storage).init(1 + ux, ux, uy)
    want = [np.array(f).reshape(-1) for f in lat.moments()]
    got = [torch.full((N,), -1.0, dtype=torch.float64, pin_memory=True).numpy() for _ in range(3)]
    assert lbm.load().lbm_read_moments(lat.h, *(g.ctypes.data for g in got)) == 0
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


def test_a_failed_read_writes_nothing():
    """Without host memory for the pageable field, the page-locked one is not written either,
    then or later. A process of its own, whose address space may not grow during the call."""
    import os
    import subprocess
    import sys
    code = """
import resource, numpy as np, torch
from paper_2607_20650_gb300 import lbm
lib = lbm.load()
N = 1 << 19
ux = np.full(N, 1e-2)
lat = lbm.Lattice(N, 1, 0.8, storage="f32").init(1 + ux, ux, ux)
rho = torch.full((N,), -1.0, dtype=torch.float64, pin_memory=True).numpy()
uxo = np.full(N, -1.0)
a, b = rho.ctypes.data, uxo.ctypes.data
torch.cuda.synchronize()
size = [int(l.split()[1]) << 10 for l in open("/proc/self/status") if l.startswith("VmSize")][0]
old = resource.getrlimit(resource.RLIMIT_AS)
resource.setrlimit(resource.RLIMIT_AS, (size, old[1]))
s = lib.lbm_read_moments(lat.h, a, b, None)
resource.setrlimit(resource.RLIMIT_AS, old)
torch.cuda.synchronize()
assert s == 2, s                                # LBM_ENOMEM
assert (rho == -1.0).all() and (uxo == -1.0).all()
assert lib.lbm_read_moments(lat.h, a, b, None) == 0
assert abs(rho - 1.01).max() < 1e-5 and abs(uxo - 1e-2).max() < 1e-5
"""
    env = dict(os.environ, GLIBC_TUNABLES="glibc.malloc.mmap_threshold=65536")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr

"""Transfers of state and moments with host memory that other calls use at the
same time: two threads restoring from one array, a transfer beside a copy from
an overlapping slice, fields that are slices of one array, and memory mapped
from a file, read-only as a source."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2607_20650_gb300 import build, lbm  # noqa: E402

NX, NY = 1023, 257          # 9 N doubles: 18.9 MB, several turns of the ring of slots
N = NX * NY


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    lbm.load()


def _state(seed):
    return (1e-2 * np.random.default_rng(seed).standard_normal((9, N))).astype(np.float32).astype(np.float64)


def _run(*jobs):
    failed = []

    def call(job):
        try:
            job()
        except BaseException as e:   # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=call, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


def test_two_threads_restore_from_one_array():
    h = _state(1)

    def job():
        lat = lbm.Lattice(NX, NY, 0.8, storage="f32", stream=torch.cuda.Stream())
        for _ in range(10):
            lat.write_populations(h)
        assert np.array_equal(lat.populations(), h)
        lat.close()

    _run(job, job)


def test_transfer_beside_a_copy_from_an_overlapping_slice():
    big = np.concatenate([_state(2).reshape(-1), np.full(N, 0.5)])
    h, tail = big[: 9 * N], big[9 * N - N // 2: 10 * N - N // 2]   # begins inside h, ends beyond it
    want = 1.0 + 0.0 * tail

    def restore():
        lat = lbm.Lattice(NX, NY, 0.8, storage="f32", stream=torch.cuda.Stream())
        for _ in range(10):
            lat.write_populations(h.reshape(9, N))
        assert np.array_equal(lat.populations().reshape(-1), h)

    def start():
        lat = lbm.Lattice(NX, NY, 0.8, storage="f32", stream=torch.cuda.Stream())
        for _ in range(10):
            lat.init(None, tail, None)
        rho, ux, _ = lat.moments()
        assert np.abs(rho.reshape(-1) - want).max() < 1e-5
        assert np.abs(ux.reshape(-1) - tail).max() < 1e-5

    _run(restore, start)


@pytest.mark.parametrize("order", [(0, 1, 2), (0, 2, 1), (2, 0, 1)])
def test_moments_into_slices_of_one_array(order):
    n = (1 << 20) + 3   # fields of more than 8 MB, off page boundaries
    r = np.random.default_rng(3)
    ux, uy = 1e-2 * r.standard_normal((2, n))
    lat = lbm.Lattice(n, 1, 0.8, storage="f32").init(1 + ux, ux, uy)
    dev = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
    lbm.lbm_moments_device(lat.h, *dev)
    want = [d.double().cpu().numpy() for d in dev]
    buf = np.full(3 * n + 2, -1.0)
    out = [buf[1 + k * n: 1 + (k + 1) * n] for k in order]
    assert lbm.load().lbm_read_moments(lat.h, *(o.ctypes.data for o in out)) == 0
    for a, b in zip(out, want):
        assert np.array_equal(a, b)
    assert buf[0] == -1.0 and buf[-1] == -1.0


@pytest.mark.parametrize("nx,ny", [(NX, NY), (2049, 1031)])   # 2049 x 1031: fields of 16.9 MB
def test_memory_mapped_files(tmp_path, nx, ny):
    n = nx * ny
    h = (1e-2 * np.random.default_rng(4).standard_normal((9, n))).astype(np.float32).astype(np.float64)
    (tmp_path / "h.bin").write_bytes(h.tobytes())
    lat = lbm.Lattice(nx, ny, 0.8, storage="f32")
    ro = np.memmap(tmp_path / "h.bin", dtype=np.float64, mode="r", shape=(9, n))
    assert lbm.load().lbm_write_populations(lat.h, ro.ctypes.data, 0) == 0
    out = np.memmap(tmp_path / "out.bin", dtype=np.float64, mode="w+", shape=(9, n))
    assert lbm.load().lbm_read_populations(lat.h, out.ctypes.data, 0) == 0
    assert np.array_equal(out, h)
    lat.step(1, moments=True)
    want = lat.moments()
    mom = np.memmap(tmp_path / "mom.bin", dtype=np.float64, mode="w+", shape=(3, n))
    assert lbm.load().lbm_read_moments(lat.h, *(m.ctypes.data for m in mom)) == 0
    for a, b in zip(mom, want):
        assert np.array_equal(a, b.reshape(-1))


def _lock(address, nbytes):
    assert int(torch.cuda.cudart().cudaHostRegister(address, nbytes, 0)) == 0


def _unlock(address):
    assert int(torch.cuda.cudart().cudaHostUnregister(address)) == 0


@pytest.mark.parametrize("pieces", [((0, 1), (-1, 1)), ((0, 8), (-8, 8)), ((0, 4),), ((-4, 4),), ((3, 5),), ((0, 16),)],
                         ids=["ends", "half and half", "head", "tail", "middle", "whole"])
def test_arrays_locked_in_pieces(pieces):
    """The caller has page-locked pieces (in sixteenths) of the arrays that state and moments go to."""
    h = _state(5)
    src = h.copy()
    out = np.full((9, N), -1.0)
    mom = np.full((3, 1 << 21), -1.0)
    lat = lbm.Lattice(NX, NY, 0.8, storage="f32")
    r = np.random.default_rng(6)
    ux = 1e-2 * r.standard_normal(mom.shape[1])
    strip = lbm.Lattice(mom.shape[1], 1, 0.8, storage="f32").init(1 + ux, ux, ux)
    want = [np.array(f).reshape(-1) for f in strip.moments()]
    locked = []
    for a in (src, out, mom[1]):
        unit = a.nbytes // 16 // 65536 * 65536   # whole pages, not a page in two pieces
        base = (a.ctypes.data + 65535) // 65536 * 65536
        for first, count in pieces:
            if count == 16:
                start, nbytes = a.ctypes.data, a.nbytes
            elif first == 0:
                start, nbytes = a.ctypes.data, base - a.ctypes.data + count * unit
            elif first < 0:
                start = base + (16 + first) * unit
                nbytes = a.ctypes.data + a.nbytes - start
            else:
                start, nbytes = base + first * unit, count * unit
            _lock(start, nbytes)
            locked.append(start)
    try:
        lib = lbm.load()
        assert lib.lbm_write_populations(lat.h, src.ctypes.data, 0) == 0
        assert lib.lbm_read_populations(lat.h, out.ctypes.data, 0) == 0
        assert lib.lbm_read_moments(strip.h, *(m.ctypes.data for m in mom)) == 0
    finally:
        for a in locked:
            _unlock(a)
    assert np.array_equal(out, h)
    for a, b in zip(mom, want):
        assert np.array_equal(a, b)

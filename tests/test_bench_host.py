"""Host-side logic of bench.py on the CPU: the max-over-ranks reduction of
the timed region on a world of two gloo ranks, and the launch accounting."""
import os
import socket

import pytest

import bench

torch = pytest.importorskip("torch")


def _free_port():
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _rank(rank, world, port, q):
    import torch.distributed as dist
    os.environ["MASTER_ADDR"] = "127.0.0.1"
    os.environ["MASTER_PORT"] = str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        q.put((rank, bench.max_over_ranks(0.5 + rank, "cpu")))
    finally:
        dist.destroy_process_group()


def test_max_over_ranks_gloo_world_2():
    import torch.multiprocessing as mp
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    port = _free_port()
    procs = [ctx.Process(target=_rank, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    for p in procs:
        p.join(120)
    assert all(p.exitcode == 0 for p in procs)
    got = dict(q.get(timeout=5) for _ in range(2))
    assert got == {0: 1.5, 1: 1.5}


def test_launch_accounting_matches_graph_blocks():
    # 64-update graphs end in one counter bump; the remainder is launched
    # directly and followed by one bump.
    assert bench.launches_for(64) == 65
    assert bench.launches_for(65) == 65 + 2
    assert bench.launches_for(1000) == 15 * 65 + 40 + 1


def test_reference_arm_json_line():
    """`bench.py --impl reference` (the FP64 oracle on the host cores) prints
    one JSON line with the contract's keys; a 3-second budget keeps it short."""
    import json
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, os.path.join(root, "bench.py"), "--impl", "reference", "--steps", "2",
                        "--warmup", "3", "--ref-seconds", "3"], capture_output=True, text=True, timeout=300,
                       cwd=root)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["metric"] == bench.METRIC and d["unit"] == "MLUPS"
    assert d["value"] > 0 and d["steps"] == 2 and d["warmup"] == 3 and d["higher_is_better"] is True
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["cpu_baseline"]["value"] == d["value"]
    assert d["config"]["workload"].startswith("porous 2048x1024") and "seed 33" in d["config"]["workload"]
    assert d["config"]["stands_in_for"] == bench.WORKLOAD
    assert d["e2e"] == {"value": d["value"], "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}


@pytest.mark.parametrize("algo,layout,storage,nx,kw,name", [
    ("nptl", "bundle", "f32", 16384, {}, "k_two_lattice<float, 1, false, false>"),
    ("lptl", "stream", "f64", 512, {}, "k_two_lattice<double, 0, true, true>"),
    ("nptl", "bundle", "f16s", 512, {}, "k_two_lattice_pair<__half, false>"),
    ("nptl", "bundle", "bf16s", 511, {}, "k_two_lattice<__nv_bfloat16, 1, false, true>"),
    ("nptl", "collision", "f32", 16384, {}, "k_two_lattice_aos<float, false>"),
    ("npol", "bundle", "f32", 16384, {"aux": 24}, "k_npol<float, 1, true>"),
    ("npol", "stream", "f32", 16384, {"l2": 1 << 27}, "k_npol<float, 0, true>"),
    ("npol", "stream", "f16s", 16384, {"l2": 1 << 27}, "k_npol<__half, 0, false>"),
    ("nsol", "bundle", "f32", 512, {"aux": 1}, "k_nsol_tma<float, 1>"),
    ("aa", "bundle", "f32", 512, {}, "k_aa<float, 1, 0|1, false> (two phases)"),
])
def test_kernel_name_has_the_template_arguments_of_the_source(algo, layout, storage, nx, kw, name):
    """The name's argument count is that of the kernel's template list in the source."""
    import argparse
    import re
    args = argparse.Namespace(algo=algo, layout=layout, storage=storage, nx=nx, ny=1024, flags=0)
    assert bench.kernel_name(args, **kw) == name
    kernel, given = re.match(r"(\w+)<(.*)>", name).groups()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with open(os.path.join(root, "paper_2607_20650_gb300", "csrc", "lbm_kernels.cuh")) as f:
        src = f.read()
    params = re.findall(r"template <([^<>]*)>\s*__global__[^;{]*?\b%s\(" % kernel, src)
    assert len(params) == 1 and len(params[0].split(",")) == len(given.split(","))

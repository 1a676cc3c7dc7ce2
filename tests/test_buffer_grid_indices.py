"""Element indices of the D3Q19 buffer grid (csrc/lbm3_kernels.cuh, Halo3), on the
host: for nodes on tile and box faces, every pull that leaves the tile must read
the element that its source node publishes, by the definition of the planes in
wide integers; also where the box's planes hold more than 2^31 nodes."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_20650_gb300", "csrc")

SOURCE = r"""
#include "lbm3_kernels.cuh"
#include <cstdio>
#include <vector>
using namespace lbm::d3;
typedef __int128 W;

// the planes by their definition
static W element(const int *n, const int *nt, const int *tile, int axis, int i, const int *at) {
    const W per[3] = {(W)n[1] * n[2], (W)n[0] * n[2], (W)n[0] * n[1]};
    W first = 0;
    for (int a = 0; a < axis; ++a) first += 10 * nt[a] * per[a];
    const int c = axis == 0 ? cx(i) : axis == 1 ? cy(i) : cz(i);
    int rank = 0;
    for (int k = 0; k < i; ++k) rank += (axis == 0 ? cx(k) : axis == 1 ? cy(k) : cz(k)) == c;
    const W in = axis == 0 ? (W)at[2] * n[1] + at[1] : axis == 1 ? (W)at[2] * n[0] + at[0] : (W)at[1] * n[0] + at[0];
    return first + ((c < 0 ? 5 : 0) + rank) * nt[axis] * per[axis] + at[axis] / tile[axis] * per[axis] + in;
}

template <bool OFF32> static int check(int nx, int ny, int nz, int tx, int ty, int tz) {
    const int n[3] = {nx, ny, nz}, tile[3] = {tx, ty, tz};
    int nt[3];
    for (int a = 0; a < 3; ++a) nt[a] = (n[a] + tile[a] - 1) / tile[a];
    std::vector<int> where[3];
    for (int a = 0; a < 3; ++a)
        for (int v : {0, 1, tile[a] - 1, tile[a], n[a] / 2 / tile[a] * tile[a], n[a] - tile[a], n[a] - 2, n[a] - 1})
            if (v >= 0 && v < n[a]) where[a].push_back(v);
    Geo3 g{};
    g.nx = nx; g.ny = ny; g.nz = nz;
    for (int x : where[0]) for (int y : where[1]) for (int z : where[2]) {
        const int p[3] = {x, y, z};
        int b[3], lo[3], hi[3];
        for (int a = 0; a < 3; ++a) {
            b[a] = p[a] / tile[a];
            lo[a] = b[a] * tile[a];
            hi[a] = (lo[a] + tile[a] < n[a] ? lo[a] + tile[a] : n[a]) - 1;
        }
        const Halo3<OFF32> H(g, nt, b, p, lo, hi);
        for (int i = 0; i < Q; ++i) {
            const int c[3] = {cx(i), cy(i), cz(i)};
            int from[3], axis = -1;
            for (int a = 2; a >= 0; --a) {
                from[a] = ((p[a] - c[a]) % n[a] + n[a]) % n[a];
                const bool crosses = (c[a] > 0 && p[a] == lo[a]) || (c[a] < 0 && p[a] == hi[a]);
                if (crosses != H.crosses(i, a)) return printf("crosses\n");
                if (crosses) axis = a;
            }
            if (axis < 0) continue;
            const W want = element(n, nt, tile, axis, i, from), got = (W)H.at(i);
            if (got != want)
                return printf("box %d x %d x %d, node %d %d %d, direction %d: %lld instead of %lld\n", nx, ny, nz, x, y, z, i,
                              (long long)got, (long long)want);
        }
    }
    return 0;
}

int main() {
    if (check<true>(5, 4, 3, 2, 2, 2) || check<false>(5, 4, 3, 2, 2, 2)) return 1;
    if (check<true>(33, 21, 17, 8, 8, 8) || check<false>(33, 21, 17, 16, 8, 4)) return 1;
    if (check<true>(64, 1, 9, 32, 1, 4) || check<false>(1, 64, 9, 1, 8, 16)) return 1;
    if (check<true>(470, 470, 510, 8, 8, 8)) return 1;                                       // 19 N just below 2^31
    if (check<false>(46400, 1, 46400, 16, 1, 16) || check<false>(1, 46400, 46400, 1, 16, 16)) return 1;
    if (check<false>(46400, 46400, 1, 16, 16, 1) || check<false>(65535, 1, 65535, 512, 1, 1)) return 1;
    return 0;
}
"""


def test_every_crossing_pull_reads_what_its_source_published(tmp_path):
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("needs nvcc")
    src, exe = tmp_path / "halo.cu", tmp_path / "halo"
    src.write_text(SOURCE)
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                        "-I", CSRC, "-I", os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"),
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout

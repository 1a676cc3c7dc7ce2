"""Launch rules that depend on the device's size, compiled for the host
(csrc/lbm_internal.h): spread_evenly() for several numbers of SMs."""
import os
import shutil
import subprocess

import pytest

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_20650_gb300")

SOURCE = r"""
#include <cuda_runtime.h>
#include "lbm_internal.h"
int main() {
    using lbm::spread_evenly;
    for (int sms : {1, 20, 132, 148, 152, 300}) {
        const unsigned full = 1536u * sms / 256;   // blocks of 256 threads that fill the SMs
        if (!spread_evenly(dim3(full), dim3(32, 8), sms) || !spread_evenly(dim3(1, 1, full), dim3(8, 8, 4), sms)) return 1;
        if (full - 1 > (unsigned)sms / 4 && spread_evenly(dim3(full - 1), dim3(256), sms)) return 2;
        if (!spread_evenly(dim3(sms / 4), dim3(256), sms) || spread_evenly(dim3(sms / 4 + 1), dim3(256), sms)) return 3;
    }
    // the same grid fills a small device and not a large one
    return spread_evenly(dim3(132 * 6), dim3(256), 132) && !spread_evenly(dim3(132 * 6), dim3(256), 152) ? 0 : 4;
}
"""


def test_spread_evenly_follows_the_number_of_sms(tmp_path):
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("needs nvcc")
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(SOURCE)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", os.path.join(PKG, "csrc"),
                        "-I", os.path.join(os.path.dirname(PKG), "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)], timeout=60).returncode == 0

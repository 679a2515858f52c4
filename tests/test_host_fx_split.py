"""Host check of the rule between the two work splits of the fixed-point FP64 hop:
one warp per hop up to one block of 32 sites per SM, whatever the device's
number of SMs.  The test compiles a host-only program against the library's
internal header.  No GPU is used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_2039_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "wd_internal.cuh"
int main() {
    int bad = 0;
    for (int sms : {1, 100, 132, 148, 152, 160})
        for (long blocks : {1l, (long)sms - 1, (long)sms, (long)sms + 1, 100000l})
            for (long vh : {32 * blocks - 31, 32 * blocks}) {
                if (blocks < 1) continue;
                if (wd::fx_one_hop_per_warp(vh, sms) != (blocks <= sms)) {
                    std::printf("%ld sites, %d SMs\n", vh, sms);
                    ++bad;
                }
            }
    return bad;
}
"""


def test_split_follows_the_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "split.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "split"
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout

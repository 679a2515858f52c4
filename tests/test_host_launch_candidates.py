"""Host check of the hop's launch candidates: the kernel of one warp per hop exists
for 4-byte and 16-bit storage only, and no other storage may be sent to it.  The
test compiles a host-only program against the library's internal header."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_2039_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "dslash.cuh"
int main() {
    using namespace wd;
    int bad = 0;
    const struct { int prec; bool half, split; } types[] = {
        {WD_F64, false, false}, {WD_F32, false, true}, {WD_F16, true, true},
        {WD_BF16, true, true}, {WD_DF64, false, false}};
    for (auto &t : types)
        for (int k = 0; k < N_DSLASH_CFG; ++k) {
            const bool want = DSLASH_CFGS[k].split ? t.split : !DSLASH_CFGS[k].stage || t.half;
            if (dslash_cfg_applies(k, t.prec) != want) {
                std::printf("candidate %d, precision %d\n", k, t.prec);
                ++bad;
            }
        }
    return bad;
}
"""


def test_candidates_of_each_storage_type(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "cand.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "cand"
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout

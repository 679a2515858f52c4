"""Host check of the rule for the fixed-point copy of an FP64 handle's links
(fx_copy_kept): no lattice that fits without the copy is refused, or left without
memory for its neighbours, because of it.

The test compiles a host-only program against the library's internal header.  No
GPU is used.
"""
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
    using namespace wd;
    const size_t GB = 1000000000ull;
    int bad = 0;
    // (sites per parity, bytes free once everything else is allocated, kept?)
    struct { long vh; size_t free_bytes; bool kept; } cases[] = {
        {128, 200 * GB, true},                       // 4^4 on an empty card
        {331776, 200 * GB, true},                    // 24^3 x 48
        {1l << 24, 180 * GB, true},                  // 64^3 x 128: 19 of 180 GB
        {1l << 24, 40 * GB, false},                  // the same on a nearly full card
        {331776, GB, false},
        {128, 0, false},
        {(1l << 28) - 64, 4000 * GB, true},          // the kernel's 32-bit offsets
        {1l << 28, 4000 * GB, false},
    };
    for (auto &c : cases) {
        const long stride = pad_stride(c.vh);
        const size_t bytes = 2 * 4 * field_bytes(WD_F64, stride, 18);
        if (fx_copy_kept(bytes, c.free_bytes, stride) != c.kept) {
            std::printf("%ld sites, %zu bytes free\n", c.vh, c.free_bytes);
            ++bad;
        }
    }
    return bad;
}
"""


def test_the_copy_leaves_room(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "copy.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "copy"
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout

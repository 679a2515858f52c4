"""Conversions between the FP64 boundary and the storage precisions.

The integer forms of the FP64 <-> FP32 and FP64 <-> double-float conversions
give the bits of the conversion instructions: a small program compiled
against the library's header walks every exponent with the mantissas where
rounding, carries and binade edges lie.  And a field that goes in and comes
out again unchanged (kappa = 0) is the input rounded to the storage type, on
lattices that end inside a block."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include "df64.cuh"
using namespace wd;
typedef unsigned long long u64;
__global__ void k_narrow(long n, const u64 *in, u64 *bad) {
    const long i = (long)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const double d = __longlong_as_double((long long)in[i]);
    if (narrow_ok(d) && __float_as_uint(narrow_double(d)) != __float_as_uint(__double2float_rn(d)))
        atomicAdd(bad, 1ull);
    const df64 s = split_double(d);
    const double a = fabs(d);
    bool ok = true;
    if (a == 0) ok = __float_as_uint(s.hi) == (unsigned)(in[i] >> 32) && s.lo == 0;
    else if (a > 1e-22 && a < 1e38) {   // nearest FP32 number, FP32 remainder
        const double r = d - (double)s.hi, t = d - (double)__double2float_rn(d);
        ok = fabs(r) == fabs(t) && s.lo == __double2float_rn(r);
    }
    if (!ok) atomicAdd(bad + 1, 1ull);
}
__global__ void k_join(long n, const uint2 *in, u64 *bad) {
    const long i = (long)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float h = __uint_as_float(in[i].x), l = __uint_as_float(in[i].y);
    const double r = (double)h + (double)l;
    if (__double_as_longlong(join_double(h, l)) != __double_as_longlong(r)) atomicAdd(bad + 2, 1ull);
    if (widen_ok(h) && __double_as_longlong(widen_float(h)) != __double_as_longlong((double)h))
        atomicAdd(bad + 3, 1ull);
}
int main() {
    std::vector<u64> d;
    const u64 half = 1ull << 28, unit = 1ull << 29, all = (1ull << 52) - 1;
    const u64 mant[] = {0, 1, half - 1, half, half + 1, unit - 1, unit, unit + half - 1, unit + half,
                        unit + half + 1, 2 * unit + half, all, all - 1, all - half, all - half + 1,
                        all - unit, 0x5A5A5A5A5A5A5, 0xA5A5A5A5A5A5A};
    for (u64 s = 0; s < 2; ++s)
        for (u64 e = 0; e < 2048; ++e)
            for (u64 m : mant) d.push_back(s << 63 | e << 52 | m);
    std::vector<uint2> f;
    const unsigned hm[] = {0, 1, 0x400000, 0x7FFFFE, 0x7FFFFF}, lm[] = {0, 1, 0x200001, 0x400000, 0x7FFFFF};
    for (unsigned s = 0; s < 4; ++s)
        for (unsigned e = 0; e < 256; ++e)
            for (unsigned a : hm)
                for (int off = 20; off < 60; ++off)
                    for (unsigned b : lm) {
                        const int el = (int)e - off;
                        const unsigned lo = el < 0 ? (off == 59 ? 0 : b) : (unsigned)el << 23 | b;
                        f.push_back(make_uint2((s & 1) << 31 | e << 23 | a, (s >> 1) << 31 | lo));
                    }
    u64 *dd, *bad, got[4];
    uint2 *df;
    cudaMalloc(&dd, d.size() * 8);
    cudaMalloc(&df, f.size() * 8);
    cudaMalloc(&bad, 32);
    cudaMemset(bad, 0, 32);
    cudaMemcpy(dd, d.data(), d.size() * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(df, f.data(), f.size() * 8, cudaMemcpyHostToDevice);
    k_narrow<<<(unsigned)((d.size() + 255) / 256), 256>>>((long)d.size(), dd, bad);
    k_join<<<(unsigned)((f.size() + 255) / 256), 256>>>((long)f.size(), df, bad);
    if (cudaMemcpy(got, bad, 32, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    std::printf("%llu %llu %llu %llu\n", got[0], got[1], got[2], got[3]);
    return 0;
}
"""


def test_integer_conversions_give_the_instructions_bits(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "conv.cu", tmp_path / "conv"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_1401_2039_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0
    assert r.stdout.split() == ["0"] * 4   # narrowing, split, join, widening


def rounded(x: np.ndarray, prec: str) -> np.ndarray:
    f = x.astype(np.float32)
    if prec == "f16":
        f = f.astype(np.float16)
    elif prec == "bf16":
        return torch.from_numpy(f).to(torch.bfloat16).to(torch.float64).numpy()
    return f.astype(np.float64)


@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 6), (4, 4, 4, 4), (10, 6, 2, 6)])
def test_a_field_passes_through_rounded_to_its_storage_type(prec, dims):
    V = syn.volume(dims)
    psi = syn.gaussian_spinor(V, 71)
    x = psi.view(np.float64).reshape(-1)
    x[:12] = [0.0, -0.0, 1.0 + 2.0**-24, 1.0 + 3 * 2.0**-24, -1.0 - 2.0**-9, 1e-40, -1e-46, 1e-310,
              2.0**-126, 2.0**-127 * (1 + 2.0**-30), 1000.0, -6e-8]
    op = WilsonDirac(dims, 0.0, prec=prec)
    op.set_gauge(torch.from_numpy(syn.su3_links(dims, eps=0.3, seed=72)).cuda())
    full = op.apply(torch.from_numpy(psi).cuda(), False).cpu().numpy()
    half = np.ascontiguousarray(psi[: V // 2])
    eo = op.apply_eo(torch.from_numpy(half).cuda(), 0, False).cpu().numpy()
    op.close()
    for got, given in ((full, psi), (eo, half)):
        v = given.view(np.float64)
        want = v if prec == "f64" else rounded(v, prec)
        assert np.array_equal(got.view(np.float64), want)

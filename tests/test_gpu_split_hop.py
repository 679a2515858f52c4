"""The hopping term with one warp per hop (launch candidate 8) rounds as the
one-thread-per-site kernels: every output is compared bitwise with candidate 0
(which the parity tests hold against the oracle), on lattices below one
32-site block, ragged, and of several blocks."""
import numpy as np
import pytest
import torch

import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac

pytestmark = pytest.mark.gpu

TWISTED = tuple(np.exp(1j * np.array([0.3, 0.0, -0.9, np.pi])))


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 2), (6, 6, 2, 4), (8, 6, 6, 10)])
def test_bitwise_equal_to_one_thread_per_site(monkeypatch, prec, recon, dims):
    U = torch.from_numpy(syn.su3_links(dims, eps=0.3, seed=61)).cuda()
    V = syn.volume(dims)
    psi = torch.from_numpy(syn.gaussian_spinor(V, 62)).cuda()
    half = psi[: V // 2].contiguous()
    runs = []
    for k in (0, 8):
        monkeypatch.setenv("WD_DSLASH_CFG", str(k))
        op = WilsonDirac(dims, 0.12, TWISTED, prec=prec, recon=recon)
        op.set_gauge(U)
        assert op.dslash_tuning()["index"] == k
        out = []
        for dagger in (False, True):
            for p in (0, 1):
                out.append(op.dslash_eo(half, p, dagger))
                op.set_twisted_mass(0.05)
                out.append(op.apply_eo(half, p, dagger))
                op.set_twisted_mass(0.0)
            out.append(op.apply(psi, dagger))
        res = op.solve(psi, tol=1e-10)   # fused norms
        out.append(res.x)
        runs.append((res.info["iters"], [o.cpu().numpy() for o in out]))
        op.close()
    for it, out in runs[1:]:
        assert it == runs[0][0]
        for a, b in zip(out, runs[0][1]):
            assert np.array_equal(a, b)

"""What wd_dslash_tuning reports of FP64 hops: the fixed-point form's launch
configuration on either side of the line between its two work splits, and the
candidates in FP64 arithmetic that WD_DSLASH_CFG forces."""
import pytest
import torch

import oracle
import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac
from parity import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (16, 2, 16, 18), (10, 10, 6, 18), (16, 16, 16, 8)])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_reported_configuration(dims, prec):
    op = WilsonDirac(dims, 0.12, (1, 1, 1, -1), prec=prec)
    if prec == "f32":
        op.set_residual_precision("f64")
    op.set_gauge(torch.from_numpy(syn.su3_links(dims, seed=91)).cuda())
    blocks = (syn.volume(dims) // 2 + 31) // 32
    wide = blocks <= torch.cuda.get_device_properties(0).multi_processor_count
    for t in [op.dslash_tuning(hi=True)] + [op.dslash_tuning()] * (prec == "f64"):
        assert t["index"] == 0 and t["block"] == (512 if wide else 128)
        assert t["min_blocks"] == (1 if wide else 5)
        assert t["sites_per_thread"] == 1 and t["stage"] == 0 and not any(t["us"])
    op.close()


@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("k", range(9))
def test_forced_candidate(monkeypatch, recon, k):
    """A hop, an operator and a solve on each FP64 candidate (those for 16-bit storage and
    the one-warp-per-hop one fall back to candidate 0), and back to the fixed-point form."""
    dims, phase = (6, 4, 2, 10), syn.workloads.APBC_T
    U = syn.su3_links(dims, eps=0.3, seed=92)
    b = syn.gaussian_spinor(syn.volume(dims), 93)
    half = syn.to_half(b, dims, 1)
    monkeypatch.setenv("WD_DSLASH_CFG", str(k))
    op = WilsonDirac(dims, 0.12, phase, prec="f64", recon=recon)
    op.set_gauge(torch.from_numpy(U).cuda())
    assert op.dslash_tuning()["index"] == (k if k < 5 else 0)
    assert op.dslash_tuning()["block"] == (256 if k == 3 else 128)
    for dagger in (False, True):
        got = op.dslash_eo(torch.from_numpy(half).cuda(), 0, dagger=dagger).cpu().numpy()
        check(got, oracle.hop_eo(half, U, dims, phase, 0, dagger), "f64", what=(recon, k, dagger))
    x = op.solve(torch.from_numpy(b).cuda(), tol=1e-12).x.cpu().numpy()
    r = b - oracle.apply(x, U, dims, 0.12, phase)
    assert (r.conj() * r).real.sum() <= (1.05e-12) ** 2 * (b.conj() * b).real.sum()
    op.close()
    monkeypatch.delenv("WD_DSLASH_CFG")
    op = WilsonDirac(dims, 0.12, phase, prec="f64", recon=recon)
    op.set_gauge(torch.from_numpy(U).cuda())
    assert op.dslash_tuning()["block"] == 512
    op.close()

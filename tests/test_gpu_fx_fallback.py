"""Sites that the fixed-point FP64 hop leaves to FP64 arithmetic: their values in
both link formats with complex boundary phases, next to sites that stay, and
what a hop of nothing else costs."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac
from parity import check

pytestmark = pytest.mark.gpu

TWISTED = tuple(np.exp(1j * np.array([0.3, 0.0, -0.9, np.pi])))


# the two work splits, one warp per hop (up to one block of 32 sites per SM) and
# one per row and sense, the latter with a ragged block
@pytest.mark.parametrize("dims", [(8, 2, 16, 18), (10, 10, 6, 18)])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("every", [True, False])
def test_values(dims, recon, every):
    U = syn.su3_links(dims, eps=0.3, seed=81)
    vh = syn.volume(dims) // 2
    psi = syn.gaussian_spinor(vh, 82)
    # below the fixed-point range everywhere, or at one site in seven
    psi = psi * np.where(every | (np.arange(vh) % 7 == 0), 2.0 ** -600, 1.0)[:, None, None]
    op = WilsonDirac(dims, 0.12, TWISTED, prec="f64", recon=recon)
    op.set_gauge(torch.from_numpy(U).cuda())
    for parity, dagger in ((0, True), (1, False)):
        got = op.dslash_eo(torch.from_numpy(psi).cuda(), parity, dagger=dagger).cpu().numpy()
        ref = oracle.hop_eo(psi, U, dims, TWISTED, parity, dagger)
        # (a power of 2, so that no square underflows)
        s = 2.0 ** 600 if every else 1.0
        check(got * s, ref * s, "f64", what=(recon, parity, dagger))
    op.close()


# A hop whose sites are all left to FP64 arithmetic against one of Gaussian fields:
# with the FP64 work shared among a site's threads it takes 3.5 times as long, with
# every thread doing its whole site 10 and 12 times.
@pytest.mark.parametrize("dims", [(16, 16, 16, 32), (8, 8, 8, 16)])
def test_cost(dims):
    op = WilsonDirac(dims, 0.12, TWISTED, prec="f64")
    op.set_gauge(torch.from_numpy(syn.su3_links(dims, eps=0.3, seed=83)).cuda())
    psi = torch.from_numpy(syn.gaussian_spinor(syn.volume(dims) // 2, 84)).cuda()
    stream = torch.cuda.ExternalStream(op.work_stream)

    def us(field):
        op.field_load(0, field)
        times = []
        for _ in range(5):
            torch.cuda.synchronize()
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(stream)
            for _ in range(20):
                op.dslash_resident(0, 1)
            b.record(stream)
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 50)
        return sorted(times)[2]

    us(psi)   # warm
    assert us(psi * 2.0 ** -600) <= 6 * us(psi)
    op.close()

"""The two work splits of the FP64 fixed-point hop, one warp per hop on lattices
of at most one 32-site block per SM and one per row and sense above: a large
lattice of the one and a small ragged one of the other over the ranges of
values that each hop's exponent can meet, against the oracle within the bound
derived in test_gpu_fx.py (per hop, so it holds for either split)."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac
from test_gpu_fx import agree, hop

pytestmark = pytest.mark.gpu


# 4608 and 5400 sites per parity: 144 blocks, and 169 of which the last is ragged
@pytest.mark.parametrize("dims", [(16, 2, 16, 18), (10, 10, 6, 18)])
@pytest.mark.parametrize("case", ["plain", "site_scales", "link_scales", "tiny", "point", "nonfinite"])
def test_ranges_of_both_splits(dims, case):
    U = syn.su3_links(dims, eps=0.3, seed=51)
    vh = syn.volume(dims) // 2
    psi = syn.gaussian_spinor(vh, 52)
    rng = np.random.default_rng(53)
    if case == "site_scales":
        psi = psi * np.exp2(rng.integers(-70, 70, size=(vh, 1, 1)))
    elif case == "link_scales":
        U = U * np.exp2(rng.integers(-75, 75, size=U.shape[:2]))[..., None, None]
    elif case == "tiny":
        psi = psi * 1e-290
    elif case == "point":
        psi = np.zeros_like(psi)
        psi[vh - 1, 2, 3] = 1.0
    elif case == "nonfinite":
        psi[vh // 2, 1, 0] = np.inf
    for p, dagger in ((0, True), (1, False)):
        got = hop(dims, U, psi, p, dagger)
        with np.errstate(invalid="ignore"):
            ref, nb = agree(got, psi, U, dims, p, dagger)
        if case == "point":
            assert (got[ref == 0] == 0).all()
        if case == "nonfinite":
            # (an extent of 2 has the same neighbour on both sides)
            assert nb.sum() == 8 - sum(L == 2 for L in dims)
            assert (~np.isfinite(got[nb]).all(axis=(1, 2))).all()


def test_norm_and_solve_above_one_block_per_sm():
    dims = (10, 10, 6, 18)
    U = syn.su3_links(dims, eps=0.3, seed=61)
    b = syn.gaussian_spinor(syn.volume(dims), 62)
    op = WilsonDirac(dims, 0.12, syn.workloads.APBC_T, prec="f64")
    op.set_gauge(torch.from_numpy(U).cuda())
    x = op.solve(torch.from_numpy(b).cuda(), tol=1e-12).x.cpu().numpy()
    op.close()
    r = b - oracle.apply(x, U, dims, 0.12, syn.workloads.APBC_T)
    assert np.linalg.norm(r) <= 1.05e-12 * np.linalg.norm(b)

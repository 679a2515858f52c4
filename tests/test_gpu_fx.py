"""The FP64 hopping term in block fixed-point arithmetic (dslash_fx.cuh) at the
edges of its range, against the oracle.

Bound per component.  Let M(x) be the largest over the eight hops of
max(1, 2 max |U|) * 2 max |psi(neighbour)|, so that a hop's block exponent
stays below 2 M.  The last place of an accumulator is at most 2^-54 M.  A hop
adds at most 5 last places (half for the rounding of the sum, 3 for the omitted
low products, 1 for the half spinor's conversion, the link's 2^-62), eight hops
40 2^-54 M; the projection rounds 6 terms per hop by 2^-53
M, 48 2^-53 M; the result once more, 2^-53 8 sqrt(3) M.  Together below 82 u M
with u = 2^-53.  The oracle's own FP64 sums (at most 9 roundings per hop on
partial sums below 6 M, and the sum over hops) stay below 150 u M.  The test
allows 256 u M.
"""
import numpy as np
import pytest
import torch

import oracle
import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac

pytestmark = pytest.mark.gpu

BOUND = 256 * 2.0 ** -53
TWISTED = tuple(np.exp(1j * np.array([0.3, 0.0, -0.9, np.pi])))


def scale_map(psi_half, U, dims, out_parity):
    """M(x) of every output site, and whether a neighbour has a non-finite entry."""
    V = syn.volume(dims)
    full = np.zeros((V, 3, 4), dtype=complex)
    full[syn.parity_sites(dims, 1 - out_parity)] = psi_half
    size = np.abs(np.stack([full.real, full.imag])).max(axis=(0, 2, 3))
    bad = ~np.isfinite(full).all(axis=(1, 2))
    link = np.maximum(1.0, 2 * np.abs(np.stack([U.real, U.imag])).max(axis=(0, 3, 4)))
    x = syn.coords(dims)
    L = np.array(dims)
    sites = syn.parity_sites(dims, out_parity)
    M, nb = np.zeros(len(sites)), np.zeros(len(sites), dtype=bool)
    for mu in range(4):
        for d in (1, -1):
            y = x[sites].copy()
            y[:, mu] = (y[:, mu] + d) % L[mu]
            lex = ((y[:, 3] * L[2] + y[:, 2]) * L[1] + y[:, 1]) * L[0] + y[:, 0]
            w = link[sites, mu] if d > 0 else link[lex, mu]
            M = np.maximum(M, np.where(bad[lex], 0.0, 2 * w * size[lex]))
            nb |= bad[lex]
    return M, nb


def hop(dims, U, psi, out_parity, dagger, recon=18, phase=TWISTED):
    op = WilsonDirac(dims, 0.12, phase, prec="f64", recon=recon)
    op.set_gauge(torch.from_numpy(U).cuda())
    got = op.dslash_eo(torch.from_numpy(psi).cuda(), out_parity, dagger=dagger).cpu().numpy()
    op.close()
    return got


def agree(got, psi, U, dims, out_parity, dagger, phase=TWISTED):
    ref = oracle.hop_eo(psi, U, dims, phase, out_parity, dagger)
    M, nb = scale_map(psi, U, dims, out_parity)
    ok = ~nb
    d = (got - ref)[ok]
    err = np.maximum(np.abs(d.real), np.abs(d.imag)).max(axis=(1, 2))
    assert (err <= BOUND * M[ok]).all(), (err / np.maximum(M[ok], 1e-300)).max() * 2.0 ** 53
    return ref, nb


# 32 sites per block: below one block, ragged, several blocks
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 2), (4, 6, 2, 10), (8, 4, 6, 10)])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dagger", [False, True])
def test_lattices(dims, recon, dagger):
    U = syn.su3_links(dims, eps=0.3, seed=11)
    for p in (0, 1):
        psi = syn.gaussian_spinor(syn.volume(dims) // 2, 12 + p)
        agree(hop(dims, U, psi, p, dagger, recon), psi, U, dims, p, dagger)


@pytest.mark.parametrize("case", ["site_scales", "component_scales", "link_scales", "tiny", "huge",
                                  "point", "zero", "unit_links"])
def test_ranges(case):
    dims, p = (6, 4, 2, 8), 1
    U = syn.su3_links(dims, eps=0.3, seed=21)
    vh = syn.volume(dims) // 2
    psi = syn.gaussian_spinor(vh, 22)
    rng = np.random.default_rng(23)
    if case == "site_scales":      # every hop raises or undercuts the accumulators' exponent
        psi = psi * np.exp2(rng.integers(-70, 70, size=(vh, 1, 1)))
    elif case == "component_scales":
        psi = psi * np.exp2(rng.integers(-70, 1, size=psi.shape))
    elif case == "link_scales":    # not SU(3): link exponents other than 0, some out of range
        U = U * np.exp2(rng.integers(-75, 75, size=U.shape[:2]))[..., None, None]
    elif case == "tiny":           # the plain FP64 sites
        psi = psi * 1e-290
    elif case == "huge":
        psi = psi * np.where(rng.random((vh, 1, 1)) < 0.3, 1e200, 1.0)
    elif case == "point":
        psi = np.zeros_like(psi)
        psi[7, 1, 2] = 1.0
    elif case == "zero":
        psi = -np.zeros_like(psi)
    else:
        U = syn.unit_links(dims)
    for dagger in (False, True):
        got = hop(dims, U, psi, p, dagger)
        ref, _ = agree(got, psi, U, dims, p, dagger)
        if case in ("point", "zero"):
            assert (got[ref == 0] == 0).all()


def test_non_finite_sites():
    dims, p = (4, 4, 6, 4), 0
    U = syn.su3_links(dims, eps=0.3, seed=31)
    psi = syn.gaussian_spinor(syn.volume(dims) // 2, 32)
    psi[5, 0, 1] = np.inf
    psi[40, 2, 3] = np.nan
    got = hop(dims, U, psi, p, False)
    with np.errstate(invalid="ignore"):
        _, nb = agree(got, psi, U, dims, p, False)
    assert nb.sum() >= 8
    assert (~np.isfinite(got[nb]).all(axis=(1, 2))).all()
    assert np.isfinite(got[~nb]).all()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 6, 2, 10)])
def test_xpay_norm_and_solve(dims):
    """The xpay epilogue with the twist (Schur operator) and the fused norms (a solve
    to a residual that needs them right), in both FP64 link formats."""
    U = syn.su3_links(dims, eps=0.3, seed=41)
    b = syn.gaussian_spinor(syn.volume(dims), 42)
    for recon in (18, 12):
        op = WilsonDirac(dims, 0.12, syn.workloads.APBC_T, prec="f64", recon=recon)
        op.set_gauge(torch.from_numpy(U).cuda())
        op.set_twisted_mass(0.05)
        half = syn.to_half(b, dims, 1)
        got = op.apply_eo(torch.from_numpy(half).cuda(), parity=1, dagger=True).cpu().numpy()
        ref = oracle.apply_eo_tm(half, U, dims, 0.12, 0.05, syn.workloads.APBC_T, 1, True)
        assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
        op.set_twisted_mass(0.0)
        x = op.solve(torch.from_numpy(b).cuda(), tol=1e-12).x.cpu().numpy()
        r = b - oracle.apply(x, U, dims, 0.12, syn.workloads.APBC_T)
        assert np.linalg.norm(r) <= 1.05e-12 * np.linalg.norm(b)
        op.close()


def test_residuals_of_a_mixed_handle():
    """set_residual_precision("f64") builds the fixed-point links of the residual side,
    before and after the gauge field is loaded."""
    dims = (4, 4, 6, 4)
    U = syn.su3_links(dims, eps=0.3, seed=51)
    half = syn.gaussian_spinor(syn.volume(dims) // 2, 52)
    ref = oracle.apply_eo(half, U, dims, 0.12, syn.workloads.APBC_T, 1)
    for late in (False, True):
        op = WilsonDirac(dims, 0.12, syn.workloads.APBC_T, prec="f32")
        if not late:
            op.set_residual_precision("f64")
        op.set_gauge(torch.from_numpy(U).cuda())
        if late:   # the loaded links went through their double-float form: 48 bits
            op.set_residual_precision("f64")
        got = op.apply_eo(torch.from_numpy(half).cuda(), parity=1, residual=True).cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
        op.set_gauge(torch.from_numpy(U).cuda())
        got = op.apply_eo(torch.from_numpy(half).cuda(), parity=1, residual=True).cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
        op.close()

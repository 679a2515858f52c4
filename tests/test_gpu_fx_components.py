"""The FP64 hopping term holds FP64 accuracy in every real component, also where
the components of a neighbourhood differ by many orders of magnitude: links that
hardly mix colours with colours of different size, spins of different size, real
parts far above imaginary ones, sites far above their neighbours.

Bound.  For a real component of the output let S be the sum over its own terms,
|link real| |spinor real|, of the eight hops (spins p and q of a projection each
on their own; the third row of 12-real links as the products it is rebuilt
from).  FP64 arithmetic rounds a term once in the projection, 4 times in a rebuilt
link element, 6 times in the product with the link, 8 times in the sum over the
hops and once in the epilogue, on partial sums below S: 20 u S with u = 2^-53.
The reference is summed in 64 or more bits.
"""
import numpy as np
import pytest
import torch

import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac

pytestmark = pytest.mark.gpu

BOUND = 20 * 2.0 ** -53
PHASE = (1, 1, 1, -1)
# row s of gamma_mu (DeGrand-Rossi) has its one entry coef[s] in column col[s]
GAMMA = (((3, 2, 1, 0), (1j, 1j, -1j, -1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
         ((2, 3, 0, 1), (1j, -1j, -1j, 1j)), ((2, 3, 0, 1), (1, 1, 1, 1)))


def sizes(z):
    """|Re z|, |Im z| as one complex array."""
    return np.abs(z.real) + 1j * np.abs(z.imag)


def times(a, b, size):
    """a b, or the sizes of its real products if size."""
    if not size:
        return a * b
    return (a.real * b.real + a.imag * b.imag) + 1j * (a.real * b.imag + a.imag * b.real)


def hop_terms(full, U, dims, dagger, recon, size):
    """H full (H^dag: dagger), or with size the sum S of every real component."""
    shape = tuple(reversed(dims))
    psi = full.reshape(shape + (3, 4)).astype(np.clongdouble)
    u = U.reshape(shape + (4, 3, 3)).astype(np.clongdouble)
    if size:
        psi, u = sizes(psi), sizes(u)
    if recon == 12:
        u = u.copy()
        a, b = u[..., 0, :], u[..., 1, :]
        for c in range(3):
            i, j = (c + 1) % 3, (c + 2) % 3
            p, q = times(a[..., i], b[..., j], size), times(a[..., j], b[..., i], size)
            u[..., 2, c] = p + q if size else np.conj(p - q)
    out = np.zeros_like(psi)
    for mu in range(4):
        ax, v = 3 - mu, u[..., mu, :, :]
        col, coef = GAMMA[mu]
        ph = 1 if size else PHASE[mu]
        for fwd in (True, False):
            edge = [slice(None)] * 6
            if fwd:
                t = np.roll(psi, -1, ax)
                edge[ax] = dims[mu] - 1
                t[tuple(edge)] *= ph
                t = sum(times(v[..., :, b, None], t[..., b, None, :], size) for b in range(3))
            else:
                w = v if size else np.conj(v)
                t = sum(times(w[..., b, :, None], psi[..., b, None, :], size) for b in range(3))
                t = np.roll(t, 1, ax)
                edge[ax] = 0
                t[tuple(edge)] *= ph
            g = t[..., list(col)]
            if size:   # an imaginary coefficient exchanges the parts
                g = g if mu % 2 else g.imag + 1j * g.real
                out += t + g
            else:
                g = g * np.array(coef, dtype=np.clongdouble)
                out += t - g if fwd != dagger else t + g
    return out.reshape(-1, 3, 4)


def fields(case, dims, seed):
    """Links (mostly the usual ones) and a full-lattice spinor of the case."""
    V = syn.volume(dims)
    rng = np.random.default_rng(seed)
    U = syn.su3_links(dims, eps=0.3, seed=seed + 1)
    psi = syn.gaussian_spinor(V, seed + 2)
    slab = syn.coords(dims)[:, 3] < 3
    spread = np.exp2([0.0, -30.0, -70.0])
    if case == "unit_colours":          # colours do not mix in the slab
        U[slab] = np.eye(3)
        psi = psi * spread[:, None]
    elif case == "near_unit_one_colour":
        U[slab] = syn.su3_links(dims, eps=1e-6, seed=seed + 3)[slab]
        psi[:, 1:] = 0
    elif case == "diagonal_colours":
        d = np.exp(1j * rng.uniform(-np.pi, np.pi, size=(int(slab.sum()), 4, 2)))
        U[slab] = 0
        for k in range(2):
            U[slab, :, k, k] = d[..., k]
        U[slab, :, 2, 2] = np.conj(d[..., 0] * d[..., 1])
        psi = psi * spread[::-1, None]
    elif case == "real_part":           # an imaginary part far below, real links in the slab
        U[slab] = syn.reunitarise(rng.standard_normal((int(slab.sum()), 4, 3, 3)) + 0j)
        psi = psi.real + 1j * 2.0 ** -40 * psi.imag
    elif case == "spins":
        psi = psi * np.exp2([0.0, -30.0, -70.0, -8.0])
    elif case == "one_spin":
        psi[..., [0, 2, 3]] = 0
    elif case == "site_scales":
        psi = psi * np.exp2(rng.integers(-70, 70, size=(V, 1, 1)))
    elif case == "all_unit":
        U[:] = np.eye(3)
        psi = psi * spread[:, None]
    else:
        assert case == "gaussian"
    return U, psi


# 2304 and 4608 sites per parity, and 5400: the two work splits (at most one block
# of 32 sites per SM, and more), the last with a ragged block
@pytest.mark.parametrize("dims", [(8, 2, 16, 18), (16, 2, 16, 18), (10, 10, 6, 18)])
@pytest.mark.parametrize("case", ["gaussian", "unit_colours", "near_unit_one_colour",
                                  "diagonal_colours", "real_part", "spins", "one_spin",
                                  "site_scales", "all_unit"])
def test_every_component_is_as_good_as_fp64(dims, case):
    U, full = fields(case, dims, 71)
    for recon, parity, dagger in ((18, 0, False), (12, 1, True)):
        op = WilsonDirac(dims, 0.12, PHASE, prec="f64", recon=recon)
        op.set_gauge(torch.from_numpy(U).cuda())
        half = syn.to_half(full, dims, 1 - parity)
        got = op.dslash_eo(torch.from_numpy(half).cuda(), parity, dagger=dagger).cpu().numpy()
        op.close()
        sites = syn.parity_sites(dims, 1 - parity)
        alone = np.zeros_like(full)
        alone[sites] = half
        out = syn.parity_sites(dims, parity)
        ref = hop_terms(alone, U, dims, dagger, recon, False)[out]
        S = hop_terms(alone, U, dims, dagger, recon, True)[out]
        d = got.astype(np.clongdouble) - ref
        assert (np.abs(d.real) <= BOUND * S.real).all() and (np.abs(d.imag) <= BOUND * S.imag).all(), \
            (case, recon, float(max((np.abs(d.real) / np.maximum(S.real, 1e-300)).max(),
                                    (np.abs(d.imag) / np.maximum(S.imag, 1e-300)).max())) * 2 ** 53)

"""The batched solver's passage between canonical right-hand sides and its
interleaved fields (groups of 12 right-hand sides, 16 sites a block), and the
deferred sums of its vector updates: numbers of right-hand sides around the
group and around the warp, with FP64 and double-float residuals, against the
same system solved alone.

Both solutions have a relative residual of at most 1e-11; the operator at
kappa = 0.1 has its spectrum within 1 +- 8 kappa, so they differ by at most
2e-11 * 1.8 / 0.2 = 1.8e-10 of the norm."""
import pytest
import torch

import synthetic as syn
from paper_1401_2039_gb300 import WilsonBatch, WilsonDirac

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,residual", [("f64", None), ("f32", "df64"), ("f32", "f64")])
@pytest.mark.parametrize("nrhs", [(1, 12), (13, 3), (25, 5), (40, 2)])
def test_batch_equals_single_solves(prec, residual, nrhs):
    shapes = [(2, 2, 2, 2), (4, 6, 2, 6)]
    ops, bs = [], []
    for k, dims in enumerate(shapes):
        op = WilsonDirac(dims, 0.1, prec=prec)
        op.set_gauge(torch.from_numpy(syn.su3_links(dims, eps=0.3, seed=80 + k)).cuda())
        if residual:
            op.set_residual_precision(residual)
        ops.append(op)
        V = syn.volume(dims)
        b = torch.stack([torch.from_numpy(syn.gaussian_spinor(V, 90 + 50 * k + j)).cuda()
                         for j in range(nrhs[k])])
        b[-1] = 0          # a point source: mostly zeros
        b[-1, V // 2, 1, 2] = 1
        bs.append(b)
    batch = WilsonBatch(ops, list(nrhs))
    xs, status, infos = batch.solve(bs, tol=1e-11)
    batch.close()
    assert status == 0
    for op, b, x in zip(ops, bs, xs):
        for j in {0, b.shape[0] // 2, b.shape[0] - 1}:
            alone = op.solve(b[j], tol=1e-11).x
            assert float((x[j] - alone).norm() / alone.norm()) < 1.8e-10
        op.close()

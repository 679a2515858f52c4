"""wd_op_set_gauge has read the caller's links when it returns: a program may then
overwrite them from any stream, whatever the handle's own stream still has to do."""
import numpy as np
import pytest
import torch

import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_links_may_be_overwritten_after_the_call(prec):
    dims = (8, 8, 8, 8)
    U = torch.from_numpy(syn.su3_links(dims, eps=0.3, seed=95)).cuda()
    half = torch.from_numpy(syn.gaussian_spinor(syn.volume(dims) // 2, 96)).cuda()
    op = WilsonDirac(dims, 0.12, (1, 1, 1, -1), prec=prec)
    op.set_gauge(U)
    ref = op.dslash_eo(half, 0).cpu().numpy()
    other = torch.cuda.Stream()
    copy = U.clone()
    with torch.cuda.stream(other):   # (loading a kernel waits for the device)
        torch.empty_like(U).zero_()
    torch.cuda.synchronize()
    torch.cuda._sleep(int(2e8))      # about 0.1 s ahead of the handle's work
    op.set_gauge(copy)
    with torch.cuda.stream(other):
        copy.zero_()
    other.synchronize()
    got = op.dslash_eo(half, 0).cpu().numpy()
    op.close()
    assert np.array_equal(got, ref)

"""What wd_dslash_tuning reports of FP64 hops: the fixed-point form's launch
configuration on either side of the line between its two work splits."""
import pytest
import torch

import synthetic as syn
from paper_1401_2039_gb300 import WilsonDirac

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

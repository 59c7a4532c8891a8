"""The launch shape that untuned programs get: bit-identical to the direct
kernel on both sides of its rule's line, and explicit block sizes or RHS per
thread that the default staging cannot serve still run."""
import numpy as np
import pytest

import lattice_inputs as li
import paper_1006_4028_gb300 as dp
from gpu_common import require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 2, 6, 4), (24, 16, 12, 12)])
@pytest.mark.parametrize("prec,c12", [("mixed_fp32", 1), ("mixed_fp32", 0), ("mixed_fp16", 1), ("mixed_bf16", 1)])
def test_default_equals_direct(dims, prec, c12):
    require_gpu()
    c = dp.dp_create(0)
    try:
        f = dp.dp_field_load(c, li.su3_links(dims, 0.4, 2), dims, -1)
        dp.dp_field_set_csw(c, f, 1.7)
        n = 12
        x = torch.randn(dp.dp_spinor_bytes(c, f, prec, n) // 4, device="cuda")
        outs = []
        for block, rpt, stages in [(64, 2, 0), (0, 0, -1), (256, 0, -1), (32, 0, -1), (0, 4, -1), (160, 2, -1)]:
            o = torch.zeros_like(x)
            dp.dp_dslash_dev(c, f, 0.3, ("cosh_t", 0.4), prec, c12, 0, x.data_ptr(), o.data_ptr(), n, block, rpt, 1,
                             stages=stages)
            torch.cuda.synchronize()
            outs.append(o)
        for o in outs[1:]:
            assert torch.equal(o, outs[0])
        # a tuned shape is not changed behind the caller's back: a block size it cannot serve stays refused
        dp.dp_tune_set(c, f, prec, c12, n, 128, 2, 6)
        with pytest.raises(dp.DpError):
            dp.dp_dslash_dev(c, f, 0.3, None, prec, c12, 0, x.data_ptr(), o.data_ptr(), n, 256, 0, 1, stages=-1)
        assert np.isfinite(float(outs[0].abs().sum()))
    finally:
        dp.dp_destroy(c)

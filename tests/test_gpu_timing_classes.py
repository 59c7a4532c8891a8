"""The timers' launch counts: an application of the FP64 Schur operator is two
operator launches (the conversion of its input belongs to the first), so a
class's time per launch is that of an operator launch."""
import numpy as np
import pytest

import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dagger", [0, 1])
@pytest.mark.parametrize("eps", [0.4, 0])  # (integer arithmetic, and the scalar kernel)
def test_two_operator_launches_an_application(eps, dagger):
    require_gpu()
    ctx = dp.dp_create(0)
    dims, n = (8, 4, 6, 4), 12
    f = dp.dp_field_load(ctx, field(dims, eps, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.0)
    x = torch.randn((12, int(np.prod(dims)) // 2, n, 2), dtype=torch.float64, device="cuda")
    y = torch.zeros_like(x)
    dp.dp_timing_reset(ctx)
    dp.dp_timing_enable(ctx, True)
    for _ in range(3):
        dp.dp_schur_dev(ctx, f, 0.15, ("cosh_t", 0.4), (0, 0, 0, 0), "fp64", 1, 0, dagger, x.data_ptr(), y.data_ptr(), n)
    launches, ms = dp.dp_timing_get(ctx, "dslash_fp64")
    dp.dp_timing_enable(ctx, False)
    assert launches == 6 and ms > 0
    dp.dp_destroy(ctx)

"""What dp_autotune reports for FP64 is the time of the operator on spinors
that are not zero: a zero neighbour costs next to nothing."""
import numpy as np
import pytest

import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 12])
def test_reported_time_is_that_of_the_operator(n):
    require_gpu()
    ctx = dp.dp_create(0)
    dims = (16, 16, 8, 16)
    f = dp.dp_field_load(ctx, field(dims, 0.4, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    x = torch.randn((12, int(np.prod(dims)) // 2, n, 2), dtype=torch.float64, device="cuda")
    y = torch.zeros_like(x)
    block, rpt, stages, ms = dp.dp_autotune(ctx, f, "fp64", 1, n)
    dp.dp_tune_set(ctx, f, "fp64", 1, n, block, rpt, stages)  # (a shape the library takes back)
    real = min(dp.dp_dslash_dev(ctx, f, 0.1, None, "fp64", 1, 0, x.data_ptr(), y.data_ptr(), n, iters=10)
               for _ in range(5))
    # the reported time is the fastest of some launches: a fifth of spread
    # between runs, and no more than that below the operator's own
    assert ms > 0.8 * real
    dp.dp_destroy(ctx)

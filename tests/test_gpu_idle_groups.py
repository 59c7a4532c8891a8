"""A serving batch whose finished groups' clover inverses are freed (a field
keeps 16 masses) while other groups still iterate: the kernels may not touch an
idle group's operands, and every served result is that of a direct solve."""
import numpy as np
import pytest

import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, slice_rel

pytestmark = pytest.mark.gpu


def test_more_masses_than_a_field_keeps():
    require_gpu()
    ctx = dp.dp_create(0)
    dims, prof, src = (8, 4, 6, 4), ("cosh_t", 0.3), (1, 0, 2, 1)
    f = dp.dp_field_load(ctx, field(dims, 0.4, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    Ms = [0.02] + [0.3 + 0.02 * k for k in range(39)]
    dp.dp_serve_start(ctx, 0, 36)
    tickets = [dp.dp_submit(ctx, f, M, prof, src, 1e-11, "mixed_fp32", 1e-9) for M in Ms]
    got = [np.asarray(dp.dp_wait(ctx, t, dims[0], timeout_s=120)[0]) for t in tickets]
    dp.dp_serve_stop(ctx, True)
    # two solves to r = 1e-11 with a per-slice residual of 1e-9: C_PP within a few times 1e-9
    for k in (0, 1, 17, 39):
        one, _, _ = dp.dp_solve_point(ctx, f, Ms[k], prof, src, 1e-11, {"prec": "mixed_fp32", "slice_tol": 1e-9}, T=dims[0],
                                      allow=())
        assert slice_rel(got[k], np.asarray(one), dims[0] - 1) < 2e-8
    dp.dp_destroy(ctx)

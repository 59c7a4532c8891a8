"""The memory a served field's batch takes is the memory the scheduler counts
for it."""
import re

import numpy as np
import pytest

import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, slice_rel

pytestmark = pytest.mark.gpu

DIMS, M, PROF, SRC = (32, 16, 16, 8), 0.5, ("cosh_t", 0.3), (1, 0, 2, 1)
# a batch's reduction scratch (2048 x 64 x 8 doubles) and its tables, which admission leaves to the slack
SMALL = 9 << 20


@pytest.fixture()
def loaded():
    require_gpu()
    ctx = dp.dp_create(0)
    f = dp.dp_field_load(ctx, field(DIMS, 0.4, 9), DIMS, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    # (a direct solve first: the mass's clover inverse belongs to the field, not to the batch)
    want, _, _ = dp.dp_solve_point(ctx, f, M, PROF, SRC, 1e-11, {"prec": "mixed_fp32", "slice_tol": 1e-9}, T=DIMS[0],
                                   allow=())
    yield ctx, f, np.asarray(want)
    dp.dp_destroy(ctx)


def served(ctx, f):
    t = dp.dp_submit(ctx, f, M, PROF, SRC, 1e-11, "mixed_fp32", 1e-9)
    return np.asarray(dp.dp_wait(ctx, t, DIMS[0], timeout_s=120)[0])


def test_bytes_in_use_cover_the_batch(loaded):
    ctx, f, want = loaded
    before = dp.dp_device_bytes(ctx)
    dp.dp_serve_start(ctx, 0, 48)
    got = served(ctx, f)
    taken, counted = dp.dp_device_bytes(ctx) - before, dp.dp_serve_stats_get(ctx)["hbm_in_use"]
    dp.dp_serve_stop(ctx, True)
    assert 0 < taken <= counted + SMALL
    assert slice_rel(got, want, DIMS[0] - 1) < 2e-8  # (two solves to a per-slice residual of 1e-9)


def test_the_smallest_budget_that_admits_a_request_serves_it(loaded):
    """The budget named in a refusal is enough, and it is kept."""
    ctx, f, want = loaded
    before = dp.dp_device_bytes(ctx)
    dp.dp_serve_start(ctx, 1, 48)
    with pytest.raises(dp.DpError) as e:
        dp.dp_submit(ctx, f, M, PROF, SRC, 1e-11, "mixed_fp32", 1e-9)
    assert e.value.status == 7
    dp.dp_serve_stop(ctx, False)
    need = int(re.search(r"\((\d+) > \d+ bytes\)", e.value.message).group(1))
    # six FP64 and nine FP32 vectors and the omega sums, 48 right-hand sides: what admission has asked for all along
    v = int(np.prod(DIMS)) // 2 * 48 * 24 * 4
    assert need == 12 * v + 9 * v + v // 8 + (1 << 20)
    dp.dp_serve_start(ctx, need, 48)
    got = served(ctx, f)
    taken = dp.dp_device_bytes(ctx) - before
    dp.dp_serve_stop(ctx, True)
    assert taken <= need + SMALL
    assert slice_rel(got, want, DIMS[0] - 1) < 2e-8

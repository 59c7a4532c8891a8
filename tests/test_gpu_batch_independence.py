"""A right-hand side's numbers depend on no other of its batch: at one batch
size (the block shapes, and so the order of the sums, follow from it), with a
mass in the same slots, other neighbours leave every bit of its result."""
import numpy as np
import pytest

import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed_fp32", "mixed_fp16", "fp64"])
@pytest.mark.parametrize("dims", [(16, 4, 4, 6), (6, 2, 4, 2)])
def test_neighbours_leave_the_bits(prec, dims):
    require_gpu()
    ctx = dp.dp_create(0)
    f = dp.dp_field_load(ctx, field(dims, 0.4, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    src, T, V = (3, 1, 2, 0), dims[0], int(np.prod(dims))
    got = []
    for Ms, profs in (([0.5, 0.1, 0.8], [("cosh_t", 0.4), ("none", 0.0), ("exp_t", 0.6)]),
                      ([0.5, 3.0, 0.05], [("cosh_t", 0.4), ("cosh_4d", 0.9), ("cosh_4d", 0.2)])):
        cpp, prop, _ = dp.dp_solve_point_multi(ctx, f, Ms, profs, src, 1e-11, {"prec": prec}, T=T, V=V, want_prop=True)
        got.append((np.asarray(cpp[0]), np.asarray(prop[0])))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
    dp.dp_destroy(ctx)

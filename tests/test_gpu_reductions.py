"""The per-RHS reductions (csrc/reduce.cuh) over the block shapes they take:
1 to 5 masses (6 to 30 RHS pairs, 64 to 16 sites a block) on lattices from
half a dozen sites per parity (one partly empty block) up, in both inner
precisions, and sums whose terms differ by many orders of magnitude."""
import numpy as np
import pytest

import lattice_inputs as li
import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, slice_rel

pytestmark = pytest.mark.gpu

MS = [0.8, 0.6, 0.5, 0.4, 0.3]


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    c = dp.dp_create(0)
    yield c
    dp.dp_destroy(c)


# C_PP per slice of solves to r = 1e-11 held to a per-slice residual of 1e-9: two such solves
# differ by a few times 1e-9 relative (C_PP is quadratic in the slice)
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 6, 2), (12, 4, 6, 4)])
@pytest.mark.parametrize("nm", [1, 3, 5])
def test_batches_of_masses(ctx, dims, nm):
    f = dp.dp_field_load(ctx, field(dims, 0.4, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    src, T = (1, 0, 1, 0), dims[0]
    out = {}
    for prec in ("mixed_fp32", "fp64"):
        o = {"prec": prec, "slice_tol": 1e-9}
        cpp, _, infos = dp.dp_solve_point_multi(ctx, f, MS[:nm], [("cosh_t", 0.4)] * nm, src, 1e-11, o, T=T, allow=())
        assert all(i["status"] == 0 and i["true_rel_residue"] < 1e-10 for i in infos)
        out[prec] = cpp
    for k in range(nm):
        one, _, _ = dp.dp_solve_point(ctx, f, MS[k], ("cosh_t", 0.4), src, 1e-11,
                                      {"prec": "fp64", "batched": 0, "slice_tol": 1e-9}, T=T, allow=())
        for prec in out:
            assert slice_rel(out[prec][k], one, T - 1) < 2e-8
    dp.dp_field_free(ctx, f)


def test_a_request_does_not_depend_on_its_batch(ctx):
    """Each RHS has its own sums: a mass solved alone and next to others of
    very different residuals gives the same bits."""
    dims = (16, 4, 4, 6)
    f = dp.dp_field_load(ctx, field(dims, 0.4, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    o = {"prec": "mixed_fp32"}
    prof = [("cosh_t", 0.4), ("none", 0.0), ("exp_t", 0.6)]
    multi, _, _ = dp.dp_solve_point_multi(ctx, f, [0.5, 0.1, 0.8], prof, (3, 1, 2, 0), 1e-11, o, T=16, allow=())
    alone, _, _ = dp.dp_solve_point(ctx, f, 0.5, prof[0], (3, 1, 2, 0), 1e-11, o, T=16, allow=())
    np.testing.assert_allclose(multi[0], alone, rtol=1e-9)
    dp.dp_field_free(ctx, f)

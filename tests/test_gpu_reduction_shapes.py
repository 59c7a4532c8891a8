"""Block shapes of csrc/reduce.cuh that batches of 12 RHS do not take: one RHS
pair (256 sites a block) and one FP64 RHS, 48 and 60 RHS (8 and 16 sites), with
one to some twenty sites a thread."""
import numpy as np
import pytest

import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, slice_rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    c = dp.dp_create(0)
    yield c
    dp.dp_destroy(c)


# tolerance as for two solves to 1e-11 with a per-slice residual of 1e-9: C_PP, quadratic in the
# slice, differs by a few times 1e-9
@pytest.mark.parametrize("dims", [(4, 2, 2, 2), (16, 8, 6, 10), (32, 16, 16, 16)])
@pytest.mark.parametrize("batched", [0, 1])
def test_one_rhs_and_twelve(ctx, dims, batched):
    f = dp.dp_field_load(ctx, field(dims, 0.3, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    T = dims[0]
    out = []
    for prec in ("mixed_fp32", "fp64"):
        cpp, _, info = dp.dp_solve_point(ctx, f, 0.5, ("cosh_t", 0.4), (1, 0, 1, 0), 1e-11,
                                         {"prec": prec, "batched": batched, "slice_tol": 1e-9}, T=T, allow=())
        assert info["status"] == 0 and info["true_rel_residue"] < 1e-10
        out.append(np.asarray(cpp))
    assert slice_rel(out[0], out[1], T - 1) < 2e-8
    dp.dp_field_free(ctx, f)


@pytest.mark.parametrize("nm", [4, 5])
def test_many_masses_on_a_wide_lattice(ctx, nm):
    dims, Ms = (32, 16, 16, 16), [0.8, 0.7, 0.6, 0.5, 0.4][:nm]
    f = dp.dp_field_load(ctx, field(dims, 0.3, 9), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    prof = [("cosh_t", 0.4)] * nm
    o = {"prec": "mixed_fp32", "slice_tol": 1e-9}
    multi, _, infos = dp.dp_solve_point_multi(ctx, f, Ms, prof, (1, 0, 1, 0), 1e-11, o, T=32, allow=())
    assert all(i["status"] == 0 and i["true_rel_residue"] < 1e-10 for i in infos)
    for k in (0, nm - 1):
        one, _, _ = dp.dp_solve_point(ctx, f, Ms[k], prof[k], (1, 0, 1, 0), 1e-11, o, T=32, allow=())
        assert slice_rel(multi[k], one, 31) < 2e-8
    dp.dp_field_free(ctx, f)

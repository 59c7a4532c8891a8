"""Sums over time slices (csrc/slice_sum.cuh) under table profiles whose time
and space factors are of opposite scale: |S'|^2 times the spatial weight
leaves FP64's range in one direction or the other although S and C_PP do not
change at all."""
import numpy as np
import pytest

import lattice_inputs as li
import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, torch

pytestmark = pytest.mark.gpu

DIMS = (4, 4, 2, 4)


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    c = dp.dp_create(0)
    yield c
    dp.dp_destroy(c)


def table(pt, px, py, pz):
    return ("table", 0.0, [np.full(L, 2.0 ** p) for L, p in zip(DIMS, (pt, px, py, pz))])


def contract(ctx, Sp, prof):
    f = dp.dp_field_load(ctx, li.unit_links(DIMS), DIMS, -1)
    x = [torch.from_numpy(np.ascontiguousarray(a).view(np.float64)).cuda() for a in dp.pack_half_spinors(Sp, DIMS)]
    got = []
    for call in (dp.dp_restore_contract_dev, dp.dp_restore_contract_noalloc):
        cpp = torch.full((1, DIMS[0]), np.nan, dtype=torch.float64, device="cuda")
        call(ctx, f, [prof], [(0, 0, 0, 0)], x[0].data_ptr(), x[1].data_ptr(), cpp.data_ptr())
        torch.cuda.synchronize()
        got.append(cpp.cpu().numpy())
    dp.dp_field_free(ctx, f)
    np.testing.assert_array_equal(got[0], got[1])
    return got[0]


# (time, x, y, z) exponents of alpha.  Powers of two scale exactly, so C_PP is
# that of the unscaled propagator to the order of the FP64 sums (1e-14 for 12 x 24 x 32 positive terms)
SCALES = [(520, -50, -50, -50), (-520, 50, 50, 50), (-540, 55, 55, 55), (560, -60, -60, -60), (450, -20, -20, -20),
          (-450, 20, 20, 20), (0, 300, -300, 0), (0, 0, 265, -265), (100, -250, -265, 420), (-100, 250, 265, -420),
          (380, 10, -10, 0), (-380, 0, 10, -10)]


@pytest.mark.parametrize("p", SCALES)
def test_contraction(ctx, p):
    S = li.random_spinor(DIMS, 12, 7)
    want = contract(ctx, S, ("none", 0.0))
    got = contract(ctx, S * 2.0 ** sum(p), table(*p))
    assert np.max(np.abs(got / want - 1)) < 1e-14


@pytest.mark.parametrize("p", [(520, -50, -50, -50), (-520, 50, 50, 50)])
def test_contraction_of_general_factors(ctx, p):
    """The same with factors that are no powers of two (per-coordinate); 1e-13:
    their products and squares are rounded in either arithmetic."""
    rng = np.random.default_rng(3)
    tabs = [2.0 ** q * rng.uniform(0.5, 2.0, L) for L, q in zip(DIMS, p)]
    al = (tabs[0][:, None, None, None] * tabs[3][None, :, None, None] * tabs[2][None, None, :, None]
          * tabs[1][None, None, None, :])
    S = li.random_spinor(DIMS, 12, 7)
    want = contract(ctx, S, ("none", 0.0))
    got = contract(ctx, S * al[None, ..., None, None], ("table", 0.0, tabs))
    assert np.max(np.abs(got / want - 1)) < 1e-13


@pytest.mark.parametrize("p", [(520, -50, -50, -50), (-520, 50, 50, 50)])
def test_per_slice_accuracy(ctx, p):
    """The per-slice norms of a solve take the same sums: a constant table
    changes neither the hops nor the outcome (C_PP of two solves held to a
    per-slice residual of 1e-9 agrees to a few times that)."""
    f = dp.dp_field_load(ctx, field(DIMS, 0.4, 9), DIMS, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    o = {"prec": "fp64", "slice_tol": 1e-9}
    want, _, _ = dp.dp_solve_point(ctx, f, 0.4, ("none", 0.0), (1, 0, 1, 0), 1e-11, o, T=DIMS[0], allow=())
    got, _, info = dp.dp_solve_point(ctx, f, 0.4, table(*p), (1, 0, 1, 0), 1e-11, o, T=DIMS[0], allow=())
    assert info["slice_residue"] <= 1e-9
    assert np.max(np.abs(got / want - 1)) < 2e-8
    dp.dp_field_free(ctx, f)

"""Restore and contract (csrc/slice_sum.cuh) where its integer sums can go
wrong: extents from 2 to 256, 1 to 5 groups (lanes of 16 to 4 sites), slices
cut into uneven shares, components and profiles over hundreds of binary
orders, zeros, infinities and NaN; the no-alloc form alike."""
import numpy as np
import pytest

import lattice_inputs as li
import oracle
import paper_1006_4028_gb300 as dp
from gpu_common import require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    c = dp.dp_create(0)
    yield c
    dp.dp_destroy(c)


def contract(ctx, dims, Sp, profs, srcs):
    f = dp.dp_field_load(ctx, li.unit_links(dims), dims, -1)
    ev, od = dp.pack_half_spinors(Sp, dims)
    x = [torch.from_numpy(np.ascontiguousarray(a).view(np.float64)).cuda() for a in (ev, od)]
    got = []
    for call in (dp.dp_restore_contract_dev, dp.dp_restore_contract_noalloc):
        cpp = torch.full((len(profs), dims[0]), np.nan, dtype=torch.float64, device="cuda")
        call(ctx, f, profs, srcs, x[0].data_ptr(), x[1].data_ptr(), cpp.data_ptr())
        torch.cuda.synchronize()
        got.append(cpp.cpu().numpy())
    dp.dp_field_free(ctx, f)
    np.testing.assert_array_equal(got[0], got[1])
    return got[0]


def wanted(dims, Sp, profs, srcs):
    out = []
    for k, (p, src) in enumerate(zip(profs, srcs)):
        al = oracle.profile_alpha(p[0], p[1], dims, src)
        out.append(oracle.contract_cpp(oracle.restore(Sp[12 * k:12 * k + 12], al, dims), dims, src[0]))
    return np.asarray(out)


PROFS = [("cosh_t", 0.4), ("cosh_4d", 0.2), ("exp_t", 0.02), ("none", 0.0), ("cosh_4d", 0.05)]


# 1e-13: the oracle's own FP64 sums of 12 x 24 x sites positive terms
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (256, 2, 2, 2), (6, 4, 10, 2), (10, 6, 4, 14), (4, 64, 2, 2)])
@pytest.mark.parametrize("ng", [1, 2, 5])
def test_extents_and_groups(ctx, dims, ng):
    Sp = li.random_spinor(dims, 12 * ng, 5)
    Sp[:, 1] = 0  # a zero slice
    srcs = [(1, 0, 1, 0)] * ng
    got, want = contract(ctx, dims, Sp, PROFS[:ng], srcs), wanted(dims, Sp, PROFS[:ng], srcs)
    on = want != 0
    assert np.max(np.abs(got[on] / want[on] - 1)) < 1e-13 and np.all(got[~on] == 0)


@pytest.mark.parametrize("p2", [-480, -380, -20, 20, 380, 480])
def test_sizes_across_the_range(ctx, p2):
    """S' = alpha S with alpha = 2^p2 everywhere (a table): S, and so C_PP, does
    not change; beyond 2^+-400 the general arithmetic answers."""
    dims = (4, 4, 2, 4)
    S = li.random_spinor(dims, 12, 7)
    tab = [np.full(L, 2.0 ** (p2 // 4)) for L in dims]
    want = contract(ctx, dims, S, [("none", 0.0)], [(0, 0, 0, 0)])
    got = contract(ctx, dims, S * 2.0 ** p2, [("table", 0.0, tab)], [(0, 0, 0, 0)])
    assert np.max(np.abs(got / want - 1)) < 1e-14


def test_components_of_very_different_sizes(ctx):
    dims = (4, 4, 2, 4)
    S = li.random_spinor(dims, 12, 7) * 2.0 ** np.random.default_rng(1).integers(-90, 90, (12, 4, 4, 2, 4, 4, 3))
    got = contract(ctx, dims, S, PROFS[1:2], [(0, 0, 0, 0)])
    want = wanted(dims, S, PROFS[1:2], [(0, 0, 0, 0)])
    assert np.max(np.abs(got / want - 1)) < 1e-13


def test_infinities_and_nan_stay_in_their_slice(ctx):
    dims = (4, 4, 2, 4)
    S = li.random_spinor(dims, 24, 7)
    good = contract(ctx, dims, S, PROFS[:2], [(0, 0, 0, 0)] * 2)
    for v in (np.inf, np.nan):
        bad = S.copy()
        bad[3, 2, 1, 1, 3, 2, 1] = v
        got = contract(ctx, dims, bad, PROFS[:2], [(0, 0, 0, 0)] * 2)
        assert not np.isfinite(got[0, 2])
        got[0, 2] = good[0, 2]
        np.testing.assert_array_equal(got, good)

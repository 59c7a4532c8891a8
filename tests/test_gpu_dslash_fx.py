"""The FP64 operator in integer arithmetic (csrc/dslash_fx.cu) where it can go
wrong: right-hand-side counts that fill its blocks unevenly, extents of 2,
profiles with and without power-of-two hop factors, Dirichlet time, spinors
whose sizes differ from site to site, zeros, and the values it hands to the
FP64 arithmetic (infinities, NaN, subnormal spinors, links that are not
unitary)."""
import numpy as np
import pytest

import lattice_inputs as li
import oracle
import paper_1006_4028_gb300 as dp
from gpu_common import field, per_site_rel, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    c = dp.dp_create(0)
    yield c
    dp.dp_destroy(c)


def load(ctx, dims, bc, seed):
    U = field(dims, 0.7, seed)
    f = dp.dp_field_load(ctx, U, dims, bc)
    dp.dp_field_set_csw(ctx, f, 1.7)
    return U, f, oracle.WilsonClover(U, dims, 1.7, bc)


# 1e-14: a site's 12 components carry about 2^-55 each on either side, plus
# the oracle's own FP64 rounding of some 1e3 operations
@pytest.mark.parametrize("dims,n", [((4, 2, 2, 2), 1), ((4, 2, 4, 6), 2), ((8, 4, 6, 4), 13), ((4, 6, 4, 2), 25),
                                    ((2, 4, 2, 6), 43), ((4, 4, 4, 4), 64)])
@pytest.mark.parametrize("prof,bc", [(("none", 0.0), 1), (("cosh_4d", 0.9), -1), (("exp_t", 0.4), 0)])
def test_hop_and_full_operator(ctx, dims, n, prof, bc):
    U, f, op = load(ctx, dims, bc, 5)
    src = (1, 0, 1, 0)
    psi = li.random_spinor(dims, n, 8)
    rng = np.random.default_rng(9)
    psi *= 2.0 ** rng.integers(-20, 20, psi.shape[:5] + (1, 1))  # sizes differ between neighbours
    psi[:, 0] = 0  # a zero time slice
    p3 = (prof[0], prof[1], src)
    for kind, ref in (("hop", op.hop(psi, p3)), ("full", op.apply(psi, 0.2, p3))):
        got = dp.dp_apply(ctx, f, kind, 0.2, prof, src, "fp64", psi)
        on = np.linalg.norm(ref.reshape(-1, 12), axis=1) > 0
        assert per_site_rel(got.reshape(-1, 12)[on], ref.reshape(-1, 12)[on]) < 1e-14
        assert np.all(got.reshape(-1, 12)[~on] == 0)
    dp.dp_field_free(ctx, f)


def schur(ctx, f, x, n, dagger=0):
    out = torch.zeros_like(x)
    dp.dp_schur_dev(ctx, f, 0.15, ("cosh_t", 0.4), (0, 0, 0, 0), "fp64", 1, 0, dagger, x.data_ptr(), out.data_ptr(), n)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("dagger", [0, 1])
def test_powers_of_two_scale_exactly(ctx, dagger):
    """Block floating point: an input times 2^k gives the output times 2^k, bit
    for bit, down to the exponents the integers take."""
    dims, n = (4, 4, 2, 4), 7
    _, f, _ = load(ctx, dims, -1, 6)
    x = torch.randn((12, 64, n, 2), dtype=torch.float64, device="cuda")
    y = schur(ctx, f, x, n, dagger)
    for k in (-600, 300):
        assert torch.equal(schur(ctx, f, x * 2.0 ** k, n, dagger), y * 2.0 ** k)
    # below the integers' range: FP64 arithmetic, the same numbers to its rounding
    k = -960
    z = schur(ctx, f, x * 2.0 ** k, n, dagger) * 2.0 ** 700 * 2.0 ** 260
    assert float((z - y).norm() / y.norm()) < 1e-14
    dp.dp_field_free(ctx, f)


def test_infinities_and_nan_reach_their_neighbours_only(ctx):
    dims, n = (8, 4, 4, 4), 3
    _, f, _ = load(ctx, dims, -1, 6)
    x = torch.randn((12, 256, n, 2), dtype=torch.float64, device="cuda")
    y = schur(ctx, f, x, n)
    for v in (float("nan"), float("inf")):
        z = x.clone()
        z[5, 40, 1, 0] = v
        w = schur(ctx, f, z, n)
        hit = ~torch.isfinite(w).all(-1).all(0)  # (site, RHS)
        assert bool(hit[40, 1]) and not bool(hit[:, 0].any()) and not bool(hit[:, 2].any())
        assert 2 <= int(hit[:, 1].sum()) <= 1 + 8 * 7
        assert torch.equal(w[:, ~hit], y[:, ~hit])
    dp.dp_field_free(ctx, f)


def test_links_that_are_not_unitary(ctx):
    dims = (4, 4, 2, 4)
    U = field(dims, 0.5, 3) * 3.0
    f = dp.dp_field_load(ctx, U, dims, -1)
    dp.dp_field_set_csw(ctx, f, 0.0)
    psi = li.random_spinor(dims, 5, 4)
    got = dp.dp_apply(ctx, f, "hop", 0.0, ("cosh_t", 0.4), None, "fp64", psi)
    ref = oracle.WilsonClover(U, dims, 0.0, -1).hop(psi, ("cosh_t", 0.4, (0, 0, 0, 0)))
    assert per_site_rel(got, ref) < 1e-14
    dp.dp_field_free(ctx, f)

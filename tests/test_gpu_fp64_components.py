"""Accuracy of the FP64 operator component by component (csrc/dslash_fx.cu):
spinors whose colours differ by many binary orders at one site, on links that
do not mix the colours (or hardly do), so that a small component of the result
stands next to a large one and is not a sum of large terms.

Bound: all truncations of the integers come to less than 2^-51 of the largest
neighbour, and a component whose terms do not add up to 2^-10 of that is left
to FP64 arithmetic, on inputs held to 2^-43: below 2^-40 an application, 2^-38
with the rounding of the reference and the sums of two."""
import numpy as np
import pytest

import lattice_inputs as li
import oracle
import paper_1006_4028_gb300 as dp
from gpu_common import field, require_gpu, torch

pytestmark = pytest.mark.gpu

DIMS = (4, 4, 6, 4)
TOL = 2.0 ** -38


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    c = dp.dp_create(0)
    yield c
    dp.dp_destroy(c)


def diagonal(shape, rng):
    a = rng.uniform(-np.pi, np.pi, shape + (2,))
    U = np.zeros(shape + (3, 3), np.complex128)
    U[..., 0, 0], U[..., 1, 1] = np.exp(1j * a[..., 0]), np.exp(1j * a[..., 1])
    U[..., 2, 2] = np.exp(-1j * a.sum(-1))
    return U


def links(kind):
    if kind == "unit":
        return li.unit_links(DIMS)
    if kind == "smooth":
        return field(DIMS, 1e-6, 4)
    if kind == "diagonal":
        return diagonal(oracle.array_shape(DIMS) + (4,), np.random.default_rng(2))
    # rough links but for the eight of one site, (2, 1, 3, 2): diagonal, or a little off it
    U, d = field(DIMS, 0.7, 5), diagonal((4, 2), np.random.default_rng(2))
    if kind == "rough, one site mixing 1e-6":
        d = d @ li.su3_links((2, 2, 2, 2), 1e-6, 3).reshape(-1, 3, 3)[:8].reshape(4, 2, 3, 3)
    t, x, y, z = 2, 1, 3, 2
    for mu in range(4):
        U[t, z, y, x, mu] = d[mu, 0]
        c = [t, x, y, z]
        c[mu] -= 1
        U[c[0], c[3], c[2], c[1], mu] = d[mu, 1]
    return U


def colour_error(got, ref, site=None):
    """Largest relative error of a site's four spins of one colour."""
    d, r = np.linalg.norm(got - ref, axis=-2), np.linalg.norm(ref, axis=-2)
    if site is not None:
        t, x, y, z = site
        d, r = d[:, t, z, y, x], r[:, t, z, y, x]
    return float(np.max(d / r))


KINDS = ["unit", "smooth", "diagonal", "rough, one site diagonal", "rough, one site mixing 1e-6"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("k", [3, 6, 11, 13, 20, 45])
@pytest.mark.parametrize("prof,bc", [(("none", 0.0), 1), (("cosh_4d", 0.3), -1)])
def test_colours_of_different_sizes(ctx, kind, k, prof, bc):
    U = links(kind)
    f = dp.dp_field_load(ctx, U, DIMS, bc)
    dp.dp_field_set_csw(ctx, f, 0.0)
    op = oracle.WilsonClover(U, DIMS, 0.0, bc)
    psi = li.random_spinor(DIMS, 5, 8) * 2.0 ** (-k * np.arange(3.0))
    site = (2, 1, 3, 2) if kind.startswith("rough") else None
    src = (1, 0, 1, 0)
    for what, ref in (("hop", op.hop(psi, prof + (src,))), ("full", op.apply(psi, 0.2, prof + (src,)))):
        got = dp.dp_apply(ctx, f, what, 0.2, prof, src, "fp64", psi)
        assert colour_error(got, ref, site) < TOL, what
    dp.dp_field_free(ctx, f)


@pytest.mark.parametrize("kind", ["unit", "smooth"])
@pytest.mark.parametrize("k", [6, 13, 40])
@pytest.mark.parametrize("dagger", [0, 1])
def test_schur_operator(ctx, kind, k, dagger):
    """The same through the intermediate vector of the Schur operator, against
    the operator on each colour by itself added up (it is linear; with one
    colour of the input non-zero nothing large stands beside anything small
    but through the links)."""
    U = links(kind)
    f = dp.dp_field_load(ctx, U, DIMS, -1)
    dp.dp_field_set_csw(ctx, f, 1.0 if kind == "unit" else 0.0)
    Vh, n = int(np.prod(DIMS)) // 2, 3
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((12, Vh, n, 2), dtype=torch.float64, device="cuda", generator=g)

    def schur(v):
        out = torch.zeros_like(v)
        dp.dp_schur_dev(ctx, f, 0.15, ("cosh_t", 0.4), (0, 0, 0, 0), "fp64", 1, 0, dagger, v.data_ptr(), out.data_ptr(), n)
        torch.cuda.synchronize()
        return out
    want, parts = torch.zeros_like(x), torch.zeros_like(x)
    for c in range(3):
        one = torch.zeros_like(x)
        one[c::3] = x[c::3] * 2.0 ** (-k * c)
        parts += one
        want += schur(one)
    got = schur(parts)
    err = (got - want).reshape(4, 3, Vh, n, 2).norm(dim=(0, 4)) / want.reshape(4, 3, Vh, n, 2).norm(dim=(0, 4))
    assert float(err.max()) < 4 * TOL
    dp.dp_field_free(ctx, f)

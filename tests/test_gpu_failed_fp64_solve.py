"""An FP64 solve that fails with a number beyond the range after it has made
progress returns its last iterate: the parity that the Schur system leaves
out satisfies its own equation, (D + A) S = eta there, as for a solve that
converged.

The operator is scaled so that the sums of squares of the inner solver lie
near the end of FP64's range (mass -4 leaves the clover term alone on the
diagonal, c_sw makes it 1e-76, and Mhat is of order 1e152); which right-hand
side leaves it, and in which round, changes from one scale to the next.  The
field is an abelian flux, gauge-transformed at random: a clover term that can
be inverted and an operator that a few iterations bring down."""
import numpy as np
import pytest

import lattice_inputs as li
import paper_1006_4028_gb300 as dp
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

NONFINITE = 5


def flux(dims, seed):
    U, _ = li.abelian_flux_links(dims, 0, 1, 1, (1.0, 1.0, -2.0))
    G = li.random_gauge_transform(dims, seed)
    for mu, axis in enumerate((0, 3, 2, 1)):
        U[..., mu, :, :] = G @ U[..., mu, :, :] @ np.conj(np.swapaxes(np.roll(G, -1, axis=axis), -1, -2))
    return U


@pytest.mark.parametrize("dims", [(4, 2, 2, 2), (4, 4, 2, 2)])
def test_the_last_iterate_is_returned(dims):
    require_gpu()
    ctx = dp.dp_create(0)
    T, V, src = dims[0], int(np.prod(dims)), (1, 0, 1, 0)
    odd = np.indices((dims[0], dims[3], dims[2], dims[1])).sum(0) % 2 == 1
    late = 0
    for seed in (1, 2):
        f = dp.dp_field_load(ctx, flux(dims, seed), dims, -1)
        for e in np.arange(-76.1, -75.5, 0.05):
            dp.dp_field_set_csw(ctx, f, 10.0 ** e)
            _, prop, info = dp.dp_solve_point(ctx, f, -4.0, ("none", 0.0), src, 1e-11,
                                              {"prec": "fp64", "inner_tol": 0.5, "max_iter": 300}, T=T, V=V,
                                              want_prop=True, allow=tuple(range(1, 12)))
            late += info["status"] == NONFINITE and info["iters_outer"] > 1
            S = prop.reshape((12, dims[0], dims[3], dims[2], dims[1], 4, 3))
            R, D = (np.linalg.norm(dp.dp_apply(ctx, f, kind, -4.0, None, src, "fp64", S)[:, odd].reshape(12, -1), axis=1)
                    for kind in ("full", "hop"))  # (the source is even)
            # A^-1 and A of a block of condition 4 and a dozen FP64 operations each
            assert np.all(R <= 1e-13 * D)
        dp.dp_field_free(ctx, f)
    assert late >= 4  # (the case the test is for did occur)
    dp.dp_destroy(ctx)

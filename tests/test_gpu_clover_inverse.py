"""The in-place Gauss-Jordan inversion of diag + C where diag + C is
indefinite, so that rows are exchanged."""
import numpy as np
import pytest

import lattice_inputs as li
import paper_1006_4028_gb300 as dp
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


# backward error of Gauss-Jordan with partial pivoting on 6x6: some tens of 2^-53 |A| |y|
@pytest.mark.parametrize("M", [-4.0, -3.9, -3.5, 0.5])
def test_inverse_with_row_exchanges(M):
    require_gpu()
    ctx = dp.dp_create(0)
    dims = (4, 4, 6, 4)
    f = dp.dp_field_load(ctx, li.su3_links(dims, 0.8, 5), dims, -1)
    dp.dp_field_set_csw(ctx, f, 1.7)
    psi = li.random_spinor(dims, 1, 2)
    y = np.asarray(dp.dp_apply(ctx, f, "clover_inv", M, None, None, "fp64", psi))
    back = (4 + M) * y + np.asarray(dp.dp_apply(ctx, f, "clover", 0.0, None, None, "fp64", y))
    site = np.abs(y).reshape(-1, 12).max(1)
    err = np.abs(back - psi).reshape(-1, 12).max(1)
    assert np.all(err < 1e-13 * (abs(4 + M) + 8) * np.maximum(site, 1.0))
    dp.dp_destroy(ctx)

"""The plain FP32 kernel's register tile at its edges: rows past a query tile, ragged point
tiles, whole and partial blocks of 16 coordinates, chunks of 32, both query layouts
(resident up to 64 padded coordinates, streamed beyond)."""
import numpy as np
import pytest

import oracle
from tests._common import mixture_inputs, tol_f32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["gaussian", "exponential"])
@pytest.mark.parametrize("d", [1, 4, 15, 16, 17, 31, 36, 64, 65, 96, 130])
@pytest.mark.parametrize("n,m", [(1, 1), (63, 9), (64, 64), (65, 65), (1300, 71)])
def test_edges(n, m, d, kernel):
    from paper_2407_07096_gb300.kde import ExactGaussianKDE
    X, Q = mixture_inputs(n + 7 * m, n, m, d)
    a = 1.0 / d
    want = oracle.kde_kernel(X, Q, a, kernel)
    _, _, kappa = oracle.kde_log(X, Q, a)
    with ExactGaussianKDE(X, a, form="simt_f32", kernel=kernel) as kde:
        got = kde.query(Q)
        # a query's sum does not depend on the batch around it (same split of the points)
        alone = np.array([kde.query(Q[i:i + 1])[0] for i in (0, m // 2, m - 1)])
    assert np.all(oracle.rel_err(got, want) <= tol_f32(kappa, d))
    assert np.all(oracle.rel_err(alone, want[[0, m // 2, m - 1]]) <= tol_f32(kappa[[0, m // 2, m - 1]], d))

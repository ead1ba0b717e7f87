"""The combine and recompute kernels behind the tensor-core form at the sizes where they
can go wrong: one to 32 lanes per query, flag counts across blocks of 256 queries, groups
of 64, the one-block and the chunked sort (4096 entries), tile indices of one and two
digits, and several instances of uneven flag counts in one launch."""
import numpy as np
import pytest

import oracle
from paper_2407_07096_gb300 import datagen as G
from tests._common import tol_tc

pytestmark = pytest.mark.gpu


def _kde(*a, **k):
    from paper_2407_07096_gb300.kde import ExactGaussianKDE
    return ExactGaussianKDE(*a, **k)


def _flagging(n, m, d, seed):
    """A mixture and a bandwidth at which the error estimate flags most queries."""
    mix = G.make_mixture(seed, 10, d, -10.0, 10.0, 1.0)
    return G.sample(mix, seed, n, "data"), G.sample(mix, seed, m, "query")


@pytest.mark.parametrize("n,m,d,a", [(3000, 1, 128, 1.0), (3000, 63, 128, 1.0), (40000, 65, 100, 1.0),
                                     (5000, 257, 64, 1.0), (3317, 4097, 128, 0.9), (70000, 5000, 32, 3.0),
                                     (2000, 9000, 16, 20.0)])
def test_recomputed_queries(n, m, d, a):
    X, Q = _flagging(n, m, d, n + m)
    sel = np.unique(np.linspace(0, m - 1, 200).astype(int))
    want = oracle.kde(X, Q[sel], a)
    _, _, kappa = oracle.kde_log(X, Q[sel], a)
    with _kde(X, a) as kde:
        got = kde.query(Q)
        flagged = kde.last_recomputed()
        again = kde.query(Q)
        assert kde.last_recomputed() == flagged
        assert flagged > 0.1 * m
        # a smaller call after a larger one, and without the check
        few = kde.query(Q[:3])
    ok = want > 1e-290
    assert np.all(oracle.rel_err(got[sel], want)[ok] <= tol_tc(kappa, d)[ok])
    assert np.array_equal(got, again)
    assert np.allclose(few, got[:3], rtol=2e-4)


@pytest.mark.parametrize("n,m", [(300, 1), (300, 300), (250000, 1), (250000, 40), (30000, 2000)])
def test_lanes_per_query(n, m):
    # ranges per query from 1 to about a thousand
    X, Q = _flagging(n, m, 6, n)
    want = oracle.kde(X, Q, 0.05) / n
    with _kde(X, 0.05, normalise=True) as kde:
        got = kde.query(Q)
    _, _, kappa = oracle.kde_log(X, Q, 0.05)
    assert np.all(oracle.rel_err(got, want) <= tol_tc(kappa, 6))


def test_uneven_instances_in_one_launch():
    import torch
    from paper_2407_07096_gb300.kde import query_batch
    sizes = [(3317, 4200, 128, 1.0), (1500, 64, 8, 0.1), (70000, 300, 32, 3.0), (900, 1, 64, 0.5), (2500, 900, 128, 1.0)]
    kdes, Qs, alone = [], [], []
    for i, (n, m, d, a) in enumerate(sizes):
        X, Q = _flagging(n, m, d, 50 + i)
        kdes.append(_kde(X, a))
        Qs.append(torch.from_numpy(Q).cuda())
        alone.append(_kde(X, a).query(Q))
    for _ in range(2):
        outs = query_batch(kdes, Qs)
        torch.cuda.synchronize()
    for k, o, w in zip(kdes, outs, alone):
        # the same bits: neither the launch settings nor the neighbours matter
        np.testing.assert_allclose(o.cpu().numpy(), w, rtol=1e-12)

"""The FP64 form's work split and its exp at the sizes where they can go wrong."""
import numpy as np
import pytest

import oracle
from tests._common import mixture_inputs

pytestmark = pytest.mark.gpu


def _kde(*a, **k):
    from paper_2407_07096_gb300.kde import ExactGaussianKDE
    return ExactGaussianKDE(*a, **k)


# queries per block are the power of two at or above m (at most 32), points per tile 16 to
# 128, coordinates come in chunks of 8
@pytest.mark.parametrize("kernel", ["gaussian", "exponential", "logistic"])
@pytest.mark.parametrize("n,m,d", [(1, 1, 1), (127, 1, 8), (129, 2, 9), (1000, 3, 7), (17, 31, 16), (4097, 33, 17),
                                   (20011, 5, 3), (333, 129, 64)])
def test_split_sizes(n, m, d, kernel):
    X, Q = mixture_inputs(n + m, n, m, d, dtype=np.float64)
    a = 1.0 / d
    _, _, kappa = oracle.kde_log(X, Q, a)
    want = oracle.kde_kernel(X, Q, a, kernel)
    with _kde(X, a, kernel=kernel) as kde:
        got = kde.query(Q)
        again = kde.query(Q)
    # a squared distance of d rounded terms, the exponent's own rounding and exp: a few
    # eps (2.2e-16) times (d + kappa)
    assert np.all(oracle.rel_err(got, want) <= 4 * 2.0 ** -52 * (8 + d + kappa))
    assert np.array_equal(got, again)


def test_sizes_change_on_one_handle():
    X, Q = mixture_inputs(5, 3001, 700, 4, dtype=np.float64)
    want = oracle.kde(X, Q, 0.3) / 3001
    with _kde(X, 0.3, normalise=True) as kde:
        for m in (700, 1, 33, 700, 7):
            assert np.all(oracle.rel_err(kde.query(Q[:m]), want[:m]) <= 1e-13)


def test_exponent_range():
    # one point at the origin, one query per exponent: normal, the last normal ones, the
    # denormal range, zero; each term is exp of an exactly known argument
    x = np.array([0.0, 1e-300, 1e-9, 0.3, 40.0, 600.0, 707.99, 708.01, 720.0, 744.0, 745.0, 746.0, 1e6])
    q = np.sqrt(x).reshape(-1, 1)
    want = np.exp(-(q[:, 0] * q[:, 0]))
    with _kde(np.zeros((1, 1)), 1.0) as kde:
        got = kde.query(q)
    normal = want > 1e-307
    assert np.all(np.abs(got[normal] - want[normal]) <= 3 * 2.0 ** -53 * want[normal])
    assert np.all(np.abs(got[~normal] - want[~normal]) <= 2 * 5e-324 + 1e-15 * want[~normal])


def test_queries_on_several_streams():
    # queued on different streams without waiting: the handle's partial sums are shared
    import torch
    X, Q = mixture_inputs(11, 60000, 96, 5, dtype=np.float64)
    with _kde(X, 0.2) as kde:
        want = [kde.query(Q + 0.1 * i) for i in range(6)]
        Qd = [torch.from_numpy(Q + 0.1 * i).cuda() for i in range(6)]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(3)]
        outs = [kde.query_dev(Qd[i], stream=streams[i % 3]) for i in range(6)]
        torch.cuda.synchronize()
    for o, w in zip(outs, want):
        assert np.array_equal(o.cpu().numpy(), w)


@pytest.mark.parametrize("kernel", ["gaussian", "exponential", "logistic"])
@pytest.mark.parametrize("n,m,d", [(60000, 96, 5), (3001, 33, 9), (20000, 1, 3), (257, 6, 17)])
def test_captured_queries_beside_others(n, m, d, kernel):
    # replays on two streams and plain queries on a third: the same bits as one at a time
    import torch
    X, Q = mixture_inputs(12, n, m, d, dtype=np.float64)
    with _kde(X, 0.2, kernel=kernel) as kde:
        want = [kde.query(Q + 0.1 * i) for i in range(3)]
        Qd = [torch.from_numpy(Q + 0.1 * i).cuda() for i in range(3)]
        graphs = [torch.cuda.CUDAGraph() for _ in range(2)]
        outs = [torch.empty(m, dtype=torch.float64, device="cuda") for _ in range(3)]
        for i in range(2):
            with torch.cuda.graph(graphs[i]):
                kde.query_dev(Qd[i], outs[i])
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(3)]
        for _ in range(4):
            for i in range(2):
                with torch.cuda.stream(streams[i]):
                    graphs[i].replay()
            kde.query_dev(Qd[2], outs[2], stream=streams[2])
        torch.cuda.synchronize()
        for o, w in zip(outs, want):
            assert np.array_equal(o.cpu().numpy(), w)

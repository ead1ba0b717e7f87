"""GPU E2LSH (Sec. 2) against the CPU oracle: hash values bit for bit (integers decided in
the same FP32 arithmetic on both sides), near-neighbour lists as exact index sets (the
result is unique: the distinct points sharing a bucket, in increasing order), edge cases,
and the pipeline into the weighted subset sums (Sec. 3.1)."""
import numpy as np
import pytest

import oracle
from tests._common import mixture_inputs

pytestmark = pytest.mark.gpu


def _cls():
    from paper_2407_07096_gb300 import build
    build.build()
    from paper_2407_07096_gb300.lsh import E2LSH
    return E2LSH


def _lists(off, idx):
    return [idx[off[j]:off[j + 1]].tolist() for j in range(len(off) - 1)]


@pytest.mark.parametrize("d", [1, 3, 16, 100])
def test_hash_values_bit_exact(d):
    import torch
    E = _cls()
    X, Q = mixture_inputs(60 + d, 3000, 200, d, spread=8.0)
    Q[:4] = np.float32(1e15) * np.sign(Q[:4] + 0.5)  # saturating values
    with E(X, 4, 10, seed=d) as lsh:
        got = lsh.hash_dev(torch.from_numpy(Q).cuda()).cpu().numpy()
        gx = lsh.hash_dev(torch.from_numpy(X).cuda()).cpu().numpy()
        A, B = lsh.A, lsh.B
    assert np.array_equal(got, oracle.lsh_hash(Q, A, B))
    assert np.array_equal(gx, oracle.lsh_hash(X, A, B))


@pytest.mark.parametrize("K,L", [(3, 8), (2, 1), (1, 63), (5, 20)])
def test_candidates_exact(K, L):
    E = _cls()
    X, Q = mixture_inputs(70 + K * L, 6000, 300, 8, spread=6.0)
    Q[::9] += np.float32(500.0)  # far queries: empty lists
    with E(X, K, L, seed=K * 100 + L) as lsh:
        off, idx = lsh.query(Q)
        A, B = lsh.A, lsh.B
    woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q, A, B), K, L)
    assert np.array_equal(off, woff)
    assert np.array_equal(idx, widx)
    assert all(len(c) == 0 for c in _lists(off, idx)[::9])


def test_device_entry_point_edges_and_identical_points():
    import torch
    E = _cls()
    X, Q = mixture_inputs(80, 2000, 64, 5)
    with E(X, 3, 6, seed=1) as lsh:
        off_h, idx_h = lsh.query(Q)
        off_d, idx_d = lsh.query_dev(torch.from_numpy(Q).cuda())
        torch.cuda.synchronize()
        assert np.array_equal(off_d.cpu().numpy(), off_h) and np.array_equal(idx_d.cpu().numpy(), idx_h)
        # caller-provided output arrays (large enough, then too small for the lists)
        ob, ib = np.full(70, -1, np.int64), np.full(len(idx_h) + 5, -1, np.int64)
        o2, i2 = lsh.query(Q, out=(ob, ib))
        assert np.array_equal(o2, off_h) and np.array_equal(i2, idx_h) and np.shares_memory(i2, ib)
        o3, i3 = lsh.query(Q, out=(ob, np.zeros(3, np.int64)))
        assert np.array_equal(o3, off_h) and np.array_equal(i3, idx_h)
        o0, i0 = lsh.query(Q[:0])
        assert o0.tolist() == [0] and len(i0) == 0
        # every data point finds itself
        off_x, idx_x = lsh.query(X[:100])
        assert all(j in c for j, c in enumerate(_lists(off_x, idx_x)))
    # all points identical: a query at that point gets every index once
    Xs = np.repeat(X[:1], 777, axis=0)
    with E(Xs, 4, 5, seed=2) as lsh:
        off, idx = lsh.query(Xs[:3])
    assert off.tolist() == [0, 777, 1554, 2331] and np.array_equal(idx[:777], np.arange(777))
    with E(X[:1], 2, 2, seed=3) as lsh:  # n = 1
        off, idx = lsh.query(X[:1])
    assert off.tolist() == [0, 1] and idx.tolist() == [0]


def test_validation():
    from paper_2407_07096_gb300 import _lib as L
    E = _cls()
    X, _ = mixture_inputs(81, 100, 1, 4)
    for K, Lt in ((0, 3), (2, 0), (2, 64)):
        with pytest.raises(L.StagKdeError) as e:
            E(X, K, Lt)
        assert e.value.code == L.EINVAL
    bad = X.copy()
    bad[3, 1] = np.nan
    with pytest.raises(L.StagKdeError):
        E(bad, 2, 2)
    with E(X, 2, 2) as lsh:
        with pytest.raises(L.StagKdeError):
            lsh.query(bad[:5])


def test_pipeline_into_subset_sums():
    # candidate lists from the tables, evaluated by the weighted subset sums
    from paper_2407_07096_gb300.kde import ExactGaussianKDE
    from tests.test_subset_gpu import _check, _kappa
    E = _cls()
    X, Q = mixture_inputs(82, 5000, 150, 6, spread=5.0)
    with E(X, 3, 10, seed=5) as lsh:
        off, idx = lsh.query(Q)
        A, B = lsh.A, lsh.B
    woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q, A, B), 3, 10)
    assert np.array_equal(off, woff) and np.array_equal(idx, widx)
    W = np.full(len(idx), 2.0, dtype=np.float32)
    with ExactGaussianKDE(X, 0.2, form="simt_f32") as kde:
        got = kde.query_subset(Q, off, idx, W)
        full = kde.query(Q)
    want = oracle.kde_subset(X, Q, 0.2, woff, widx, W)
    _check(got, want, _kappa(X, Q, 0.2, woff, widx, W, "gaussian"), 6)
    assert np.all(got <= 2.0 * full * (1 + 1e-5))  # a subset of the points, weight 2


@pytest.mark.slow
def test_sort_path_beyond_the_bitmap():
    # n above what the shared-memory bitmap path serves (2^22 points): repeats across
    # tables are removed by the radix-sort path instead; the lists are the same
    E = _cls()
    r = np.random.default_rng(17)
    X = r.normal(scale=40.0, size=(4_500_000, 2)).astype(np.float32)
    Q = r.normal(scale=40.0, size=(40, 2)).astype(np.float32)
    with E(X, 4, 3, seed=17) as lsh:
        off, idx = lsh.query(Q)
        A, B = lsh.A, lsh.B
    woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q, A, B), 4, 3)
    assert woff[-1] > 1000
    assert np.array_equal(off, woff)
    assert np.array_equal(idx, widx)


@pytest.mark.slow
def test_bitmap_slices_and_duplicates():
    # n spanning two slices of the bitmap path (at most 1572864 points each), with every
    # point repeated three times (identical hash values: the same buckets)
    E = _cls()
    r = np.random.default_rng(18)
    base = r.normal(scale=6.0, size=(600_000, 3)).astype(np.float32)
    X = np.concatenate([base, base[::-1], base])
    Q = np.concatenate([base[:30], r.normal(scale=6.0, size=(30, 3)).astype(np.float32)])
    with E(X, 3, 4, seed=18) as lsh:
        off, idx = lsh.query(Q)
        A, B = lsh.A, lsh.B
    woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q, A, B), 3, 4)
    assert np.array_equal(off, woff)
    assert np.array_equal(idx, widx)
    lists = _lists(off, idx)
    for j in range(30):  # a data point finds all three copies of itself
        assert {j, len(X) - 600_000 + j, 2 * 600_000 - 1 - j} <= set(lists[j])


@pytest.mark.slow
def test_paper_parameters_sampled():
    # the paper's example tables (K = 6, L = 50) over 200000 points, 2000 queries; 40 lists
    # checked against the oracle
    from paper_2407_07096_gb300 import datagen as G
    E = _cls()
    X, Q = G.workload_single_d16(4, n=200_000, m=2000)
    with E(X, 6, 50, seed=9) as lsh:
        off, idx = lsh.query(Q)
        A, B = lsh.A, lsh.B
    rows = np.random.default_rng(5).choice(len(Q), 40, replace=False)
    woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q[rows], A, B), 6, 50)
    got = _lists(off, idx)
    want = _lists(woff, widx)
    for r, w in zip(rows, want):
        assert got[r] == w


def test_membership_is_exact_when_keys_collide(monkeypatch):
    # With 12-bit bucket keys (a test hook; the library uses 58 bits) many different
    # K-tuples share a key: the build must pick a salt under which no two tuples of the
    # points share a key, and each lookup must reject a run whose tuple differs from the
    # query's. Tight data (few tuples per table) and far queries (new tuples only):
    # hundreds of lookups land on another tuple's key, and the lists must still equal
    # the oracle's, which compares tuples.
    E = _cls()
    rng = np.random.default_rng(5)
    X = (0.3 * rng.normal(size=(3000, 8))).astype(np.float32)
    near = (0.3 * rng.normal(size=(2000, 8))).astype(np.float32)
    far = rng.uniform(-200, 200, size=(20000, 8)).astype(np.float32)
    Q = np.concatenate([near, far])
    monkeypatch.setenv("STAG_KDE_LSH_KEY_BITS", "12")
    with E(X, 3, 8, seed=11) as lsh:
        off, idx = lsh.query(Q)
        A, B = lsh.A, lsh.B
    monkeypatch.delenv("STAG_KDE_LSH_KEY_BITS")
    HX, HQ = oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q, A, B)
    woff, widx = oracle.lsh_candidates(HX, HQ, 3, 8)
    assert np.array_equal(off, woff)
    assert np.array_equal(idx, widx)
    assert off[len(near)] > 0  # the near queries found their buckets
    # the far queries' tuples are new: count the lookups whose 12-bit key space alone
    # would have matched a bucket (distinct tuples per table vs 4096 keys)
    tuples = sum(len({tuple(r) for r in HX[:, l * 3:(l + 1) * 3]}) for l in range(8))
    assert tuples * len(far) / 4096 > 100


@pytest.mark.parametrize("n,m", [(5, 3), (17, 40), (131072, 2), (131073, 200), (884000, 2), (890000, 30)])
def test_one_pass_lists_at_their_limits(n, m):
    # key directories of 0 and more bits; with and without the summary bitmap, every block
    # size, lists at fixed and at measured offsets; both ways to fetch them
    import torch
    r = np.random.default_rng(n)
    X = (r.standard_normal((n, 3)) * 6).astype(np.float32)
    Q = np.concatenate([X[r.integers(0, n, m - 1)] + np.float32(0.1), np.full((1, 3), 1e6, np.float32)])
    with _cls()(X, 3, 7, seed=2) as lsh:
        woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, lsh.A, lsh.B), oracle.lsh_hash(Q, lsh.A, lsh.B), 3, 7)
        off, idx = lsh.query_dev(torch.from_numpy(Q).cuda())
        hoff, hidx = lsh.query(Q)
    assert np.array_equal(off.cpu().numpy(), woff) and np.array_equal(idx.cpu().numpy(), widx)
    assert np.array_equal(hoff, woff) and np.array_equal(hidx, widx)


@pytest.mark.parametrize("m1", [40, 2000])  # lists at fixed and at measured offsets (m n 4 above 256 MB)
@pytest.mark.parametrize("then", ["other stream", "host", "fetch on two streams"])
def test_a_queued_fetch_is_not_overtaken_by_the_next_query(m1, then):
    # the copy of the kept lists is queued behind 50 ms of other work on its stream; a query
    # with other rows, on another stream, comes before it has run
    import ctypes
    import torch
    from paper_2407_07096_gb300 import _lib
    n, lib = 100_000, _lib.load()
    r = np.random.default_rng(m1)
    X = (r.standard_normal((n, 3)) * 6).astype(np.float32)
    Q1 = torch.from_numpy(X[r.integers(0, n, m1)] + np.float32(0.1)).cuda()
    Q2 = torch.from_numpy(X[r.integers(0, n, 33)] - np.float32(0.2)).cuda()
    with _cls()(X, 3, 7, seed=4) as lsh:
        want = [t.cpu().numpy() for Q in (Q1, Q2) for t in lsh.query_dev(Q)]
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        off, total = torch.empty(m1 + 1, dtype=torch.int64, device="cuda"), ctypes.c_int64()
        torch.cuda.synchronize()
        _lib.check(lib.stag_lsh_query_dev(lsh._h, Q1.data_ptr(), m1, off.data_ptr(), None, 0, ctypes.byref(total),
                                          a.cuda_stream))
        idx = [torch.full((total.value,), -7, dtype=torch.int64, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        with torch.cuda.stream(a):
            torch.cuda._sleep(100_000_000)
        _lib.check(lib.stag_lsh_fetch_dev(lsh._h, idx[0].data_ptr(), total.value, a.cuda_stream))
        if then == "fetch on two streams":
            _lib.check(lib.stag_lsh_fetch_dev(lsh._h, idx[1].data_ptr(), total.value, b.cuda_stream))
        with torch.cuda.stream(b):
            got2 = lsh.query(Q2.cpu().numpy()) if then == "host" else lsh.query_dev(Q2)
        torch.cuda.synchronize()
    assert np.array_equal(off.cpu().numpy(), want[0]) and np.array_equal(idx[0].cpu().numpy(), want[1])
    if then == "fetch on two streams":
        assert np.array_equal(idx[1].cpu().numpy(), want[1])
    got2 = [np.asarray(t.cpu() if isinstance(t, torch.Tensor) else t) for t in got2]
    assert np.array_equal(got2[0], want[2]) and np.array_equal(got2[1], want[3])


def test_captured_fetch():
    import ctypes
    import torch
    from paper_2407_07096_gb300 import _lib
    lib = _lib.load()
    X, Q = mixture_inputs(83, 4000, 90, 4)
    with _cls()(X, 3, 6, seed=6) as lsh:
        woff, widx = lsh.query(Q)
        Qd = torch.from_numpy(Q).cuda()
        off, total = torch.empty(91, dtype=torch.int64, device="cuda"), ctypes.c_int64()
        idx = torch.zeros(len(widx), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        _lib.check(lib.stag_lsh_query_dev(lsh._h, Qd.data_ptr(), 90, off.data_ptr(), None, 0, ctypes.byref(total), None))
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            _lib.check(lib.stag_lsh_fetch_dev(lsh._h, idx.data_ptr(), total.value,
                                              torch.cuda.current_stream().cuda_stream))
        g.replay()
        torch.cuda.synchronize()
    assert np.array_equal(idx.cpu().numpy(), widx) and np.array_equal(off.cpu().numpy(), woff)


@pytest.mark.parametrize("copies", [1, 20])  # up to one query per SM (1024 threads each), and more
@pytest.mark.parametrize("n,L", [(300, 1), (2049, 1), (3000, 63), (140_000, 5), (890_000, 3)])
def test_large_buckets(n, L, copies):
    # one function per table: buckets of about a third of the points, far more members than the
    # threads load ahead (8 each of 256, 512 and 1024), over one or many tables
    import torch
    r = np.random.default_rng(n)
    X = r.standard_normal((n, 2)).astype(np.float32) * 3
    Q = np.concatenate([X[:5] + np.float32(0.01), np.full((1, 2), 1e6, np.float32), X[5:8]])
    Q = np.concatenate([Q + np.float32(0.3 * i) for i in range(copies)])
    with _cls()(X, 1, L, seed=3) as lsh:
        woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, lsh.A, lsh.B), oracle.lsh_hash(Q, lsh.A, lsh.B), 1, L)
        off, idx = lsh.query_dev(torch.from_numpy(Q).cuda())
    assert np.array_equal(off.cpu().numpy(), woff) and np.array_equal(idx.cpu().numpy(), widx)


@pytest.mark.parametrize("m", [60, 1500])  # lists at fixed and at measured offsets
@pytest.mark.parametrize("way", ["host", "host with room", "device"])
def test_lists_without_room_for_the_32_bit_copy(m, way, monkeypatch):
    # each allocation of a first query fails in turn: those that the two-pass kernels can do
    # without are done without, the others report out of memory; the next query is unharmed
    import torch
    from paper_2407_07096_gb300 import _lib as L
    n = 60_000
    r = np.random.default_rng(m)
    X = (r.standard_normal((n, 3)) * 5).astype(np.float32)
    Q = X[r.integers(0, n, m)] + np.float32(0.1)
    answered = 0
    for k in range(1, 8):
        with _cls()(X, 3, 5, seed=9) as lsh:
            if k == 1:
                woff, widx = oracle.lsh_candidates(oracle.lsh_hash(X, lsh.A, lsh.B), oracle.lsh_hash(Q, lsh.A, lsh.B),
                                                   3, 5)
                room = (np.empty(m + 1, np.int64), np.empty(len(widx), np.int64))

            def query():
                if way == "device":
                    return [t.cpu().numpy() for t in lsh.query_dev(torch.from_numpy(Q).cuda())]
                return lsh.query(Q, out=room) if way == "host with room" else lsh.query(Q)
            monkeypatch.setenv("STAG_KDE_INJECT_ALLOC_FAIL", str(k))
            try:
                off, idx = query()
                assert np.array_equal(off, woff) and np.array_equal(idx, widx), k
                answered |= 1 << k
            except L.StagKdeError as e:
                assert e.code == L.ENOMEM, (k, e)
            finally:
                monkeypatch.delenv("STAG_KDE_INJECT_ALLOC_FAIL")
            off, idx = query()
            assert np.array_equal(off, woff) and np.array_equal(idx, widx), k
    # device: scratch, then the 32-bit lists; host: queries, scratch, the 32-bit lists, the lists
    for k in ((2,) if way == "device" else (3, 4)):
        assert answered >> k & 1, (k, bin(answered))


@pytest.mark.parametrize("K,d", [(1, 3), (9, 7), (33, 4), (40, 2)])
@pytest.mark.parametrize("m", [60, 3242, 3243])  # a warp per lookup up to 9728 of them (L = 3), then a thread
def test_lookup_forms(K, d, m, monkeypatch):
    # fewer and more functions than lanes; with 9-bit keys, lookups that land on another
    # tuple's key must be rejected by comparing the functions
    import torch
    r = np.random.default_rng(K * 10 + m)
    X = (r.standard_normal((600, d)) * (0.5 if K > 9 else 0.15)).astype(np.float32)
    near = X[r.integers(0, 600, m // 2)]
    far = (r.uniform(-100, 100, size=(m - len(near), d))).astype(np.float32)
    Q = np.concatenate([near, far])
    A, B = (r.standard_normal((3 * K, d)) * 0.3).astype(np.float32), (4 * r.random(3 * K)).astype(np.float32)
    HX, HQ = oracle.lsh_hash(X, A, B), oracle.lsh_hash(Q, A, B)
    tuples = max(len({tuple(v) for v in HX[:, l * K:(l + 1) * K]}) for l in range(3))
    if tuples <= 12:  # (few enough for a salt that keeps them apart)
        monkeypatch.setenv("STAG_KDE_LSH_KEY_BITS", "9")
    with _cls()(X, K, 3, A=A, B=B) as lsh:
        off, idx = lsh.query_dev(torch.from_numpy(Q).cuda())
    woff, widx = oracle.lsh_candidates(HX, HQ, K, 3)
    assert woff[len(near)] > 0
    assert np.array_equal(off.cpu().numpy(), woff) and np.array_equal(idx.cpu().numpy(), widx)

"""What a user of this library has it do, as cases that a timing program can prepare and run.

The cases go through the public entry points (`ExactGaussianKDE.query`, `.query_dev`,
`.query_subset_dev`, `.degrees`, `query_batch`, `E2LSH.query_dev`) at the sizes of the
package's own workloads (benchmark, serving, paper shapes) and at ragged ones between
them. Inputs are Gaussian mixtures like the workloads': means uniform in [-10, 10]^d
(or [-5, 5]^2 for the FP64 one), unit or log-uniform standard deviations, queries from
the same mixture, made on the GPU from the seed alone. The library takes its point set
from host memory, so `prepare` brings it there and builds the handle, as a program does
once per data set.
"""
import math

import numpy as np
import torch

from paper_2407_07096_gb300 import kde as K
from paper_2407_07096_gb300 import lsh as H


def listed():
    return [
        # FP64 data, the plain method's size (n = m = 1000, d = 2): host arrays in and out.
        dict(name="f64_n1000_m1000_d2", kind="query", host=True, dtype="f64", form="auto", kernel="gaussian",
             n=1000, m=1000, d=2, comps=3, spread=5.0, a=1.0),
        # The smallest request a server or an interactive program makes: one query against
        # a small data set, host array in, one density out.
        dict(name="host_m1_n10000_d4", kind="query", host=True, dtype="f32", form="auto", kernel="gaussian",
             n=10000, m=1, d=4, comps=10, spread=10.0, a=0.25),
        # A typical served request (m log-uniform in [1, 4096], its median) on a mid-sized
        # resident data set, host arrays.
        dict(name="host_m61_n207031_d32", kind="query", host=True, dtype="f32", form="auto", kernel="gaussian",
             n=207031, m=61, d=32, comps=10, spread=10.0, a=1.0 / 32),
        # A small device batch on the largest served data set: reading the points dominates.
        dict(name="dev_m17_n2000000_d128", kind="query", host=False, dtype="f32", form="auto", kernel="gaussian",
             n=2000000, m=17, d=128, comps=10, spread=10.0, a=1.0 / 128),
        # The benchmark's single instance.
        dict(name="dev_m100000_n100000_d16", kind="query", host=False, dtype="f32", form="auto", kernel="gaussian",
             n=100000, m=100000, d=16, comps=10, spread=10.0, a=0.1),
        # The large workload's point set (50 components of unequal width), a quarter of its
        # queries.
        dict(name="dev_m25000_n2000000_d64", kind="query", host=False, dtype="f32", form="auto", kernel="gaussian",
             n=2000000, m=25000, d=64, comps=50, spread=10.0, a=0.05),
        # The widest tensor-core operands, a real data set's ragged n and d.
        dict(name="dev_m10000_n1193514_d100", kind="query", host=False, dtype="f32", form="auto", kernel="gaussian",
             n=1193514, m=10000, d=100, comps=10, spread=10.0, a=0.01),
        # d beyond the tensor-core form (28 x 28 images): the plain FP32 form.
        dict(name="dev_m10000_n70000_d784", kind="query", host=False, dtype="f32", form="auto", kernel="gaussian",
             n=70000, m=10000, d=784, comps=10, spread=10.0, a=1.0 / 784),
        # The exponential kernel function (always the plain FP32 form).
        dict(name="exp_m100000_n100000_d16", kind="query", host=False, dtype="f32", form="auto", kernel="exponential",
             n=100000, m=100000, d=16, comps=10, spread=10.0, a=0.3),
        # Many instances of uneven n, m, d and a in one batched call.
        dict(name="batch_256", kind="batch", instances=256, nlo=1000, nhi=200000, mlo=64, mhi=8192),
        # Candidate lists of hash tables (K = 6, L = 50) over a million points, summed over by
        # the subset sums: the inner step of a hashing-based estimator.
        dict(name="lsh_m10000_n1000000_d16", kind="lsh", n=1000000, m=10000, d=16, comps=10, spread=10.0,
             K=6, L=50, a=0.1),
        # The random-sampling estimator: 1000 weighted points per query.
        dict(name="subset_m100000_n1000000_d16", kind="subset", n=1000000, m=100000, d=16, comps=10, spread=10.0,
             a=0.1, per=1000, kernel="gaussian"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["request", "request", "device", "device", "device", "plain", "f64", "batch", "lsh", "subset",
                       "degrees"])
    if kind == "request":
        d = _log_int(rng, 2, 128)
        return dict(kind="query", host=True, dtype="f32", form="auto", kernel="gaussian",
                    n=_log_int(rng, 10000, 2000000), m=_log_int(rng, 1, 4096), d=d, comps=10, spread=10.0, a=1.0 / d)
    if kind == "device":
        d = _log_int(rng, 2, 128)
        n = _log_int(rng, 10000, 2000000)
        m = _log_int(rng, 1, max(1, min(100000, 10 ** 10 // n)))
        return dict(kind="query", host=False, dtype="f32", form="auto", kernel="gaussian", n=n, m=m, d=d,
                    comps=rng.choice([10, 50]), spread=10.0, a=rng.choice([0.1, 1.0, 2.0]) / d)
    if kind == "plain":
        d = _log_int(rng, 2, 784)
        n = _log_int(rng, 1000, 200000)
        m = _log_int(rng, 1, max(1, min(100000, 10 ** 11 // (n * (d + 4)))))
        return dict(kind="query", host=False, dtype="f32", form="simt_f32",
                    kernel=rng.choice(["gaussian", "exponential", "logistic"]), n=n, m=m, d=d, comps=10, spread=10.0,
                    a=1.0 / d)
    if kind == "f64":
        d = _log_int(rng, 1, 64)
        n = _log_int(rng, 200, 100000)
        m = _log_int(rng, 1, max(1, min(10000, 10 ** 9 // (n * (d + 8)))))
        return dict(kind="query", host=rng.random() < 0.5, dtype="f64", form="auto",
                    kernel=rng.choice(["gaussian", "gaussian", "exponential", "logistic"]), n=n, m=m, d=d, comps=3,
                    spread=5.0, a=1.0 / d)
    if kind == "batch":
        return dict(kind="batch", instances=rng.randint(5, 96), nlo=1000, nhi=_log_int(rng, 20000, 200000), mlo=64,
                    mhi=_log_int(rng, 512, 8192))
    if kind == "lsh":
        return dict(kind="lsh", n=_log_int(rng, 20000, 2000000), m=_log_int(rng, 64, 10000), d=rng.randint(4, 48),
                    comps=10, spread=10.0, K=rng.choice([6, 8]), L=rng.randint(8, 50), a=0.1)
    if kind == "subset":
        per = _log_int(rng, 30, 3000)
        return dict(kind="subset", n=_log_int(rng, 10000, 1000000), m=_log_int(rng, 100, min(100000, 10 ** 8 // per)),
                    d=_log_int(rng, 2, 128) if per < 1000 else rng.choice([2, 5, 8, 16]), comps=10, spread=10.0, a=0.1,
                    per=per, kernel=rng.choice(["gaussian", "gaussian", "exponential"]))
    return dict(kind="degrees", n=_log_int(rng, 2000, 100000), d=_log_int(rng, 2, 64), comps=10, spread=10.0, a=0.1)


# ------------------------------------------------------------------ inputs
def _mixture(g, count, means, stds, dtype):
    """count rows on the GPU: component uniform, unit normal noise times its width."""
    comps, d = means.shape
    out = torch.empty((count, d), dtype=dtype, device="cuda")
    step = max(1, (1 << 26) // d)
    for r in range(0, count, step):
        c = min(step, count - r)
        k = torch.randint(comps, (c,), generator=g, device="cuda")
        z = torch.randn((c, d), generator=g, device="cuda", dtype=dtype)
        out[r:r + c] = means[k] + stds[k, None] * z
    return out


def _points(case, seed, n, m, d, comps, spread, dtype=torch.float32):
    """(X, Q) on the GPU: the data set and the queries of one mixture."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + n * 7 + m * 3 + d)
    means = spread * (2.0 * torch.rand((comps, d), generator=g, device="cuda", dtype=dtype) - 1.0)
    if comps >= 50:  # unequal widths, log-uniform in [0.5, 2]
        stds = torch.exp(math.log(0.5) + math.log(4.0) * torch.rand(comps, generator=g, device="cuda", dtype=dtype))
    else:
        stds = torch.ones(comps, device="cuda", dtype=dtype)
    return _mixture(g, n, means, stds, dtype), _mixture(g, m, means, stds, dtype)


def _inputs(case, seed):
    dtype = torch.float64 if case.get("dtype") == "f64" else torch.float32
    return _points(case, seed, case["n"], case.get("m", 1), case["d"], case["comps"], case["spread"], dtype)


def _batch_inputs(case, seed):
    """Per instance: (X, Q, a)."""
    r = np.random.RandomState(1)
    cnt = case["instances"]
    ns = np.exp(r.uniform(math.log(case["nlo"]), math.log(case["nhi"]), cnt)).astype(int)
    ms = np.exp(r.uniform(math.log(case["mlo"]), math.log(case["mhi"]), cnt)).astype(int)
    aa = r.uniform(0.01, 1.0, cnt)
    for i in range(cnt):
        d = (8, 32, 128)[i % 3]
        X, Q = _points(case, seed * 1009 + i, int(ns[i]), int(ms[i]), d, 10, 10.0)
        yield X, Q, float(aa[i])


def _subset_lists(case, seed):
    """Ragged per-query lists around `per` entries: offsets, indices, weights n / length."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 13)
    m, per, n = case["m"], case["per"], case["n"]
    if per == 1000:  # every query draws the same number of samples
        ln = torch.full((m,), per, dtype=torch.int64, device="cuda")
    else:
        ln = torch.randint(0, 2 * per, (m,), generator=g, device="cuda")
    off = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ln, 0, out=off[1:])
    total = int(off[-1])
    idx = torch.randint(n, (total,), generator=g, device="cuda")
    w = torch.repeat_interleave(n / ln.clamp(min=1).float(), ln)
    return off, idx, w


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    if case["kind"] == "batch":
        kdes, Qs, a0, b0 = [], [], 0, []
        for X, Q, a in _batch_inputs(case, seed):
            kdes.append(K.ExactGaussianKDE(X.cpu().numpy(), a))
            Qs.append(Q)
            b0.append((a0, a0 + Q.shape[0]))
            a0 += Q.shape[0]
        flat = torch.empty(a0, dtype=torch.float64, device="cuda")  # one result vector, a slice per instance
        return dict(kind="batch", kdes=kdes, Qs=Qs, flat=flat, outs=[flat[u:v] for u, v in b0])
    X, Q = _inputs(case, seed)
    if case["kind"] == "lsh":
        Xh = X.cpu().numpy()
        return dict(kind="lsh", lsh=H.E2LSH(Xh, case["K"], case["L"], seed=seed), Q=Q,
                    kde=K.ExactGaussianKDE(Xh, case["a"], form="simt_f32"))
    if case["kind"] == "subset":
        kde = K.ExactGaussianKDE(X.cpu().numpy(), case["a"], form="simt_f32", kernel=case["kernel"])
        off, idx, w = _subset_lists(case, seed)
        return dict(kind="subset", kde=kde, Q=Q, off=off, idx=idx, w=w)
    if case["kind"] == "degrees":
        return dict(kind="degrees", kde=K.ExactGaussianKDE(X.cpu().numpy(), case["a"]))
    kde = K.ExactGaussianKDE(X.cpu().numpy(), case["a"], form=case["form"], kernel=case["kernel"])
    return dict(kind="query", kde=kde, host=case["host"], Q=Q.cpu().numpy() if case["host"] else Q)


def run(state):
    if state["kind"] == "batch":
        K.query_batch(state["kdes"], state["Qs"], state["outs"])
        return state["flat"]
    if state["kind"] == "lsh":
        off, idx = state["lsh"].query_dev(state["Q"])
        return [off, state["kde"].query_subset_dev(state["Q"], off, idx)]
    if state["kind"] == "subset":
        return state["kde"].query_subset_dev(state["Q"], state["off"], state["idx"], state["w"])
    if state["kind"] == "degrees":
        return state["kde"].degrees()
    return state["kde"].query(state["Q"]) if state["host"] else state["kde"].query_dev(state["Q"])


# ------------------------------------------------------------------ what a pass cannot do without
def _batch_sizes(case):
    r = np.random.RandomState(1)
    cnt = case["instances"]
    ns = np.exp(r.uniform(math.log(case["nlo"]), math.log(case["nhi"]), cnt)).astype(int)
    ms = np.exp(r.uniform(math.log(case["mlo"]), math.log(case["mhi"]), cnt)).astype(int)
    return [(int(ns[i]), int(ms[i]), (8, 32, 128)[i % 3]) for i in range(cnt)]


def work(case):
    """Points, queries and lists read once, results written once; per pair the d subtractions
    and d multiply-adds of the squared distance and one kernel function value (counted 1)."""
    if case["kind"] == "batch":
        s = _batch_sizes(case)
        return {"bytes": sum((n + m) * d * 4 + m * 8 for n, m, d in s),
                "flops": sum(n * m * (3 * d + 1) for n, m, d in s)}
    n, m, d = case["n"], case.get("m", case["n"]), case["d"]
    if case["kind"] == "lsh":
        # hash values of the queries, the offsets and the sums; at these settings a query has
        # about 0.4 % of the points as candidates: their indices written and read, a point's
        # row and a kernel value each
        e = m * n // 250
        return {"bytes": m * d * 4 + case["K"] * case["L"] * (d + 1) * 4 + m * 16 + e * 16 + n * d * 4,
                "flops": 2 * m * d * case["K"] * case["L"] + e * (3 * d + 2)}
    if case["kind"] == "subset":
        e = m * case["per"]
        return {"bytes": e * 12 + (n + m) * d * 4 + m * 16, "flops": e * (3 * d + 2)}
    if case["kind"] == "degrees":
        return {"bytes": n * d * 4 + n * 8, "flops": n * n * (3 * d + 1)}
    es = 8 if case["dtype"] == "f64" else 4
    return {"bytes": (n + m) * d * es + m * 8, "flops": n * m * (3 * d + 1)}


# ------------------------------------------------------------------ 64-bit values
def _kernel64(d2, a, kernel):
    if kernel == "gaussian":
        return torch.exp(-a * d2)
    x = a * d2.sqrt()
    if kernel == "exponential":
        return torch.exp(-x)
    t = torch.exp(-x)
    return 4.0 * t / (1.0 + t) ** 2


def _dist2_64(Q, X):
    if X.shape[1] <= 8:
        d2 = torch.zeros((Q.shape[0], X.shape[0]), dtype=torch.float64, device="cuda")
        for k in range(X.shape[1]):
            d2 += (Q[:, k, None] - X[None, :, k]) ** 2
        return d2
    q2, x2 = (Q * Q).sum(1), (X * X).sum(1)
    return torch.addmm(q2[:, None] + x2[None, :], Q, X.T, alpha=-2.0).clamp_(min=0.0)


def _sums64(X, Q, a, kernel):
    X, Q = X.double(), Q.double()
    c = X.mean(0)  # smaller magnitudes, so the cancellation below costs no visible digits
    X, Q = X - c, Q - c
    out = torch.zeros(Q.shape[0], dtype=torch.float64, device="cuda")
    qs, xs = 4096, 65536
    for i in range(0, Q.shape[0], qs):
        for j in range(0, X.shape[0], xs):
            out[i:i + qs] += _kernel64(_dist2_64(Q[i:i + qs], X[j:j + xs]), a, kernel).sum(1)
    return out


def exact(case, seed):
    if case["kind"] == "lsh":
        return None
    if case["kind"] == "batch":
        return torch.cat([_sums64(X, Q, a, "gaussian") for X, Q, a in _batch_inputs(case, seed)])
    X, Q = _inputs(case, seed)
    if case["kind"] == "degrees":
        return _sums64(X, X, case["a"], "gaussian")
    if case["kind"] == "subset":
        off, idx, w = _subset_lists(case, seed)
        out = torch.zeros(case["m"], dtype=torch.float64, device="cuda")
        X, Q = X.double(), Q.double()
        rows = torch.repeat_interleave(torch.arange(case["m"], device="cuda"), off[1:] - off[:-1])
        step = max(1, (1 << 27) // case["d"])
        for s in range(0, idx.numel(), step):
            r, i = rows[s:s + step], idx[s:s + step]
            d2 = ((Q[r] - X[i]) ** 2).sum(1)
            out.index_add_(0, r, _kernel64(d2, case["a"], case["kernel"]) * w[s:s + step].double())
        return out
    got = _sums64(X, Q, case["a"], case["kernel"])
    return got.cpu().numpy() if case["host"] else got

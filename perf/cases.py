"""The work a user has this library do, as timed cases.

Every case goes through the public binding (paper_2403_18766_gb300.native)
with the workload shapes, sample-size policies and budgets of the repository's
benchmark and tests: whole fits (Algorithm 1), several fits batched into one
launch per round, a burst of served jobs, the full-data assignment in exact
and in BF16 form, and the step calls (Lloyd, sample + gather + K-means++).
Data are Gaussian mixtures drawn on the device from the seed; the centroids of
the assignment cases are a few plain torch Lloyd updates on a subsample, i.e.
what a short fit hands to the assignment.
"""
import math

import numpy as np
import torch

from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture_device

DEV = "cuda"


def listed():
    return [
        # Algorithm 1 end to end on a toy data set: 4 workers, samples of 250
        # to 2000 rows, 20 rounds; latency of the rounds is everything.
        dict(name="fit_10k_n2_k5", kind="fit", m=10_000, n=2, k=5, workers=4, passes=10, rounds=20,
             s_min=250, s_max=2000, size_set=True, outliers=0.0, eval_full=False),
        # The benchmark's headline workload: 16 competing workers, samples of
        # 1,000 to 64,000 rows, f(C, X) after each round.
        dict(name="fit_1m_n16_k25", kind="fit", m=1_000_000, n=16, k=25, workers=16, passes=10, rounds=4,
             s_min=1000, s_max=64_000, size_set=False, outliers=0.0, eval_full=True),
        # Three groups of workers with different k over the same rows (64
        # workers in all), every round in one launch; the samples exceed L2.
        dict(name="batch_4m_n32_k10_25_50", kind="batch", m=4_000_000, n=32, ks="10,25,50", workers="22,21,21",
             passes=10, rounds=1, s_min=2000, s_max=131_072, outliers=0.01),
        # A large data set clustered in fast mode: the rows are packed to BF16
        # inside the call and the labels come from the tensor cores.
        dict(name="fit_fast_10m_n64_k100", kind="fit_fast", m=10_000_000, n=64, k=100, workers=8, passes=4,
             rounds=1, s_min=20_000, s_max=60_000, outliers=0.0),
        # A burst of jobs of different shapes, FP32 and BF16 storage, served
        # from pinned host memory with four running at once.
        dict(name="serve_burst_6", kind="serve", jobs=6, shapes=1, m=1_000_000, workers=16, passes=10, rounds=3,
             outliers=0.005),
        # Labelling a handful of new rows with known centroids.
        dict(name="assign_2k_n3_k4", kind="assign", m=2_000, n=3, k=4, outliers=0.0, labels=True),
        # Labels and f(C, X) of the headline workload's rows.
        dict(name="assign_1m_n16_k25", kind="assign", m=1_000_000, n=16, k=25, outliers=0.0, labels=True),
        # Odd width, odd row count, k between tile sizes.
        dict(name="assign_1m5_n21_k33", kind="assign", m=1_500_007, n=21, k=33, outliers=0.01, labels=True),
        # The largest exact assignment: 2.56 GB of rows, 100 centroids.
        dict(name="assign_10m_n64_k100", kind="assign", m=10_000_000, n=64, k=100, outliers=0.0, labels=True),
        # The same rows held packed in BF16 by the caller, close calls
        # re-scored in FP32 (tau = 1e-3).
        dict(name="bf16_10m_n64_k100", kind="assign_bf16", m=10_000_000, n=64, k=100, tau=1e-3, certified=False,
             outliers=0.0),
        # Lloyd's iterations alone on one large sample.
        dict(name="lloyd_131k_n32_k50", kind="lloyd", m=131_072, n=32, k=50, max_iter=300, tol=1e-4, outliers=0.01),
        # Drawing a sample, gathering it and seeding K-means++ on it.
        dict(name="seed_64k_of_4m_n32_k50", kind="seed", m=4_000_000, s=64_000, n=32, k=50, trials=3,
             outliers=0.01),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "batch", "fit_fast", "serve", "assign", "assign", "assign", "assign_bf16",
                       "assign_bf16", "lloyd", "lloyd", "seed"])
    if kind == "fit":
        m = _log_int(rng, 10_000, 2_000_000)
        n = rng.choice([2, 3, 5, 8, 13, 16, 24, 32])
        s_max = _log_int(rng, 2_000, min(64_000, m))
        return dict(kind="fit", m=m, n=n, k=rng.randint(3, 50), workers=rng.choice([2, 4, 8, 16]),
                    passes=rng.choice([4, 10]), rounds=rng.randint(1, 5),
                    s_min=max(100, s_max // rng.choice([4, 16, 64])), s_max=s_max, size_set=rng.random() < 0.3, outliers=rng.choice([0.0, 0.01]),
                    eval_full=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="batch", m=_log_int(rng, 200_000, 4_000_000), n=rng.choice([8, 16, 20, 32]),
                    ks="%d,%d" % (rng.randint(5, 20), rng.randint(21, 50)),
                    workers="%d,%d" % (rng.randint(4, 20), rng.randint(4, 20)), passes=rng.choice([3, 6, 10]), rounds=1,
                    s_min=2000, s_max=_log_int(rng, 8_000, 131_072), outliers=rng.choice([0.0, 0.01]))
    if kind == "fit_fast":
        return dict(kind="fit_fast", m=_log_int(rng, 500_000, 8_000_000), n=rng.choice([24, 32, 48, 61, 64]),
                    k=rng.randint(20, 100), workers=rng.choice([4, 8]), passes=rng.choice([2, 4]), rounds=1,
                    s_min=10_000, s_max=_log_int(rng, 20_000, 60_000), outliers=0.0)
    if kind == "serve":
        return dict(kind="serve", jobs=rng.randint(2, 6), shapes=rng.randint(2, 10_000),
                    m=_log_int(rng, 100_000, 1_000_000), workers=rng.choice([4, 16]), passes=rng.choice([4, 10]), rounds=rng.randint(1, 3), outliers=0.005)
    if kind == "assign":
        n = rng.randint(2, 64)
        return dict(kind="assign", m=_log_int(rng, 2_000, 6_000_000), n=n, k=_log_int(rng, 2, 128),
                    outliers=rng.choice([0.0, 0.01]), labels=rng.random() < 0.8)
    if kind == "assign_bf16":
        return dict(kind="assign_bf16", m=_log_int(rng, 100_000, 8_000_000), n=rng.choice([16, 31, 32, 50, 64]),
                    k=rng.randint(10, 200), tau=rng.choice([0.0, 1e-3, 1e-3]), certified=rng.random() < 0.4,
                    outliers=rng.choice([0.0, 0.01]))
    if kind == "lloyd":
        n = rng.choice([2, 4, 7, 16, 25, 32, 64])
        return dict(kind="lloyd", m=_log_int(rng, 1_000, 131_072), n=n, k=rng.randint(3, 64),
                    max_iter=rng.choice([20, 300]), tol=1e-4, outliers=rng.choice([0.0, 0.01]))
    m = _log_int(rng, 50_000, 4_000_000)
    return dict(kind="seed", m=m, s=_log_int(rng, 1_000, 64_000 if m > 128_000 else m // 2),
                n=rng.choice([2, 8, 15, 16, 32, 64]), k=rng.randint(3, 64), trials=rng.choice([1, 3]),
                outliers=rng.choice([0.0, 0.01]))


def _rows(case, k, seed):
    return gaussian_mixture_device(case["m"], case["n"], k, seed, outliers=case["outliers"], device=DEV)


def _centroids(X, k, seed, steps=6, sample=16_384):
    """k centroids after a few plain Lloyd updates on a subsample (deterministic: the
    member sums are one-hot products)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 77)
    S = X[torch.randint(0, X.shape[0], (sample,), generator=g, device=DEV)].double()
    C = S[torch.randperm(sample, generator=g, device=DEV)[:k]].clone()
    for _ in range(steps):
        d = (C * C).sum(1)[None, :] - 2.0 * (S @ C.T)
        one = torch.nn.functional.one_hot(d.argmin(1), k).double()
        cnt = one.sum(0)
        C = torch.where(cnt[:, None] > 0, (one.T @ S) / cnt.clamp(min=1)[:, None], C)
    return C.float().contiguous()


def _policy(case, workers, k):
    lo, hi = max(case["s_min"], 2 * k), max(case["s_max"], 2 * k)
    if case.get("size_set"):
        return native.make_policy(sizes=sorted({lo, (lo + hi) // 4 + lo // 2, (lo + hi) // 2, hi}), workers=workers,
                                  passes=case["passes"])
    return native.make_policy(s_min=lo, s_max=hi, workers=workers, passes=case["passes"],
                              kind=1 if case["kind"] == "batch" else 0)


def _ints(text):
    return [int(v) for v in text.split(",")]


def prepare(case, seed):
    kind, st = case["kind"], dict(case=case, seed=int(seed))
    if kind in ("fit", "fit_fast"):
        st["X"] = _rows(case, case["k"], seed)
        st["policy"] = _policy(case, case["workers"], case["k"])
        st["budget"] = native.make_budget(rounds=case["rounds"], eval_full_each_round=case.get("eval_full", False))
    elif kind == "batch":
        st["X"] = _rows(case, max(_ints(case["ks"])), seed)
        st["fits"] = [(k, _policy(case, w, k), native.make_budget(rounds=case["rounds"]))
                      for k, w in zip(_ints(case["ks"]), _ints(case["workers"]))]
    elif kind == "serve":
        rs = np.random.RandomState(case["shapes"])     # the jobs' shapes belong to the case, their rows to the seed
        jobs = []
        for i in range(case["jobs"]):
            # job sizes down to a tenth of the largest, the stream's widths and k
            m = int(case["m"] * 10.0 ** -rs.uniform(0.0, 1.0)) if i else case["m"]
            n, k = int(rs.choice([8, 32, 64])), int(rs.choice([5, 10, 25, 100]))
            X = gaussian_mixture_device(m, n, 2 * k, int(seed) + 31 * i, outliers=case["outliers"], device=DEV)
            Xh = torch.empty((m, n), dtype=torch.float32, pin_memory=True)
            Xh.copy_(X)
            pol = native.make_policy(s_min=max(1000, 2 * k), s_max=min(64_000, m), workers=case["workers"],
                                     passes=case["passes"])
            jobs.append((Xh, k, pol, native.make_budget(rounds=case["rounds"]), int(seed) + i, bool(i % 2)))
        st["jobs"] = jobs
    elif kind in ("assign", "assign_bf16"):
        X = _rows(case, case["k"], seed)
        st["C"] = _centroids(X, case["k"], seed)
        st["X"] = native.PackedBF16(X) if kind == "assign_bf16" else X
    elif kind == "lloyd":
        st["X"] = _rows(case, case["k"], seed)
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed) + 5)
        st["C"] = st["X"][torch.randperm(case["m"], generator=g, device=DEV)[:case["k"]]].contiguous()
    elif kind == "seed":
        st["X"] = _rows(case, case["k"], seed)
        st["C"] = torch.zeros((case["k"], case["n"]), device=DEV)
        st["deg"] = torch.ones(case["k"], dtype=torch.uint8, device=DEV)
    else:
        raise ValueError(kind)
    return st


def _fit_out(C, Y, rep):
    return dict(C=C, labels=Y, f=rep["f_full"], s_opt=rep["s_opt"], best=rep["best_worker"])


def run(state):
    c, seed = state["case"], state["seed"]
    kind = c["kind"]
    if kind == "fit":
        return _fit_out(*native.fit(state["X"], c["k"], state["policy"], state["budget"], seed=seed))
    if kind == "fit_fast":
        return _fit_out(*native.fit_dt(state["X"], c["k"], state["policy"], state["budget"], seed=seed,
                                       mode=native.BM_MODE_FAST))
    if kind == "batch":
        sess = [native.FitSession(state["X"], k, pol, bud, seed=seed + k) for k, pol, bud in state["fits"]]
        try:
            native.rounds_batch(sess, c["rounds"])
            return [_fit_out(*s.finish()) for s in sess]
        finally:
            for s in sess:
                s.close()
    if kind == "serve":
        ctx = native.ServeContext(64 << 30, max_active=4)
        try:
            ids = [ctx.submit(X, k, pol, bud, seed=s, bf16=bf16) for X, k, pol, bud, s, bf16 in state["jobs"]]
            done = [ctx.wait(i) for i in ids]
            return [dict(status=d["status"], C=d["C"], labels=d["labels"], f=d["f_full"], s_opt=d["s_opt"])
                    for d in done]
        finally:
            ctx.close()
    if kind == "assign":
        Y, f, rep = native.assign(state["X"], state["C"], labels=c["labels"])
        return dict(labels=Y, f=f) if c["labels"] else dict(f=f)
    if kind == "assign_bf16":
        Y, f, rep = native.assign_bf16(state["X"], state["C"], tau=c["tau"], certified=c["certified"])
        return dict(labels=Y, f=f)
    if kind == "lloyd":
        C, f, iters, empty = native.lloyd(state["X"], state["C"], max_iter=c["max_iter"], tol=c["tol"])
        return dict(C=C, f=f, iters=iters, empty=empty.to(torch.uint8))
    idx = native.sample(seed, native.RNG_PASS, 0, 0, 0, c["m"], c["s"])
    S = native.gather(state["X"], idx)
    return dict(idx=idx, S=S, C=native.kmeanspp(S, state["C"], state["deg"], c["trials"], seed, 0, 0, 0))


def work(case):
    """Bytes: rows read once, labels and centroids written once.  Flops: the distance
    contraction 2 n k per row of the full pass and of each pass's least two assignments."""
    kind = case["kind"]

    def fit_work(m, n, k, w, p, t, s_mean, full=1):
        rows = t * w * (p + 1) * s_mean                        # sampled rows of the rounds
        return 4 * n * (m + rows) + 4 * m, 2 * n * k * (full * m + 2 * t * w * p * s_mean)

    if kind in ("fit", "fit_fast"):
        s = (case["s_min"] + case["s_max"]) / 2
        b, f = fit_work(case["m"], case["n"], case["k"], case["workers"], case["passes"], case["rounds"], s,
                        1 + (case["rounds"] if case.get("eval_full") else 0))
    elif kind == "batch":
        s = (case["s_max"] - case["s_min"]) / max(1.0, math.log(case["s_max"] / case["s_min"]))
        parts = [fit_work(case["m"], case["n"], k, w, case["passes"], case["rounds"], s)
                 for k, w in zip(_ints(case["ks"]), _ints(case["workers"]))]
        b, f = sum(x[0] for x in parts), sum(x[1] for x in parts)
    elif kind == "serve":
        m = case["m"] * (1 + 0.39 * (case["jobs"] - 1))       # mean of 10^-U(0, 1) is 0.39
        s = (1000 + min(64_000, case["m"])) / 2
        b, f = fit_work(m, 35, 35, case["workers"] * case["jobs"], case["passes"], case["rounds"], s)
    elif kind in ("assign", "assign_bf16"):
        row = (4 * case["n"] if kind == "assign" else 2 * case["n"] + 4) + (4 if case.get("labels", True) else 0)
        b, f = case["m"] * row + 4 * case["n"] * case["k"], 2 * case["m"] * case["n"] * case["k"]
    elif kind == "lloyd":
        b, f = 4 * case["m"] * case["n"], 4 * case["m"] * case["n"] * case["k"]
    else:
        b = case["s"] * (8 + 8 * case["n"])
        f = case["s"] * case["n"] * 3 * case["k"] * case["trials"]
    return {"bytes": int(b), "flops": int(f)}


def _f64(X, C, chunk=1 << 18):
    """f(C, X) in 64 bits."""
    C = C.double()
    total = 0.0
    for i in range(0, X.shape[0], chunk):
        x = X[i:i + chunk].double()
        j = ((C * C).sum(1)[None, :] - 2.0 * (x @ C.T)).argmin(1)
        total += float(((x - C[j]) ** 2).sum())
    return total


def _lloyd64(S, C, max_iter, tol):
    S, C = S.double(), C.double()
    k, f_prev, it = C.shape[0], 0.0, 0
    while True:
        j = ((C * C).sum(1)[None, :] - 2.0 * (S @ C.T)).argmin(1)
        f = float(((S - C[j]) ** 2).sum())
        if it >= max_iter or (it and f_prev - f <= tol * f_prev):
            return C, f
        one = torch.nn.functional.one_hot(j, k).double()
        cnt = one.sum(0)
        C = torch.where(cnt[:, None] > 0, (one.T @ S) / cnt.clamp(min=1)[:, None], C)
        f_prev, it = f, it + 1


def exact(case, seed):
    kind = case["kind"]
    if kind == "assign" or kind == "assign_bf16":
        X = _rows(case, case["k"], seed)
        f = _f64(X, _centroids(X, case["k"], seed))
        return dict(labels=None, f=f) if case.get("labels", True) else dict(f=f)
    if kind == "lloyd":
        st = prepare(case, seed)
        C, f = _lloyd64(st["X"], st["C"], case["max_iter"], case["tol"])
        return dict(C=C, f=f, iters=None, empty=None)
    return None        # a fit's or a seeding's centroids depend on the library's random streams

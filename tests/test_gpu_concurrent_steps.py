"""Step calls from several threads, each on a stream of its own: the results are those of one call at
a time, and the calls share the device instead of waiting for one another."""
import threading
import time

import pytest
import torch

from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture_device

pytestmark = pytest.mark.gpu


def _jobs(s, n, k, count):
    jobs = []
    for t in range(count):
        S = gaussian_mixture_device(s, n, k, 11 + t)
        jobs.append((S, S[:k].clone(), torch.ones(k, dtype=torch.uint8, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    return jobs


def _kpp(job):
    S, C, deg, st = job
    with torch.cuda.stream(st):
        return native.kmeanspp(S, C, deg, 3, 5, 0, 0, 0)


def _lloyd(job):
    S, C, deg, st = job
    with torch.cuda.stream(st):
        return native.lloyd(S, C, max_iter=30, tol=0.0)


def _together(fn, jobs, reps):
    out, errors = [None] * len(jobs), []

    def work(i):
        try:
            for _ in range(reps):
                out[i] = fn(jobs[i])
        except Exception as e:                   # noqa: BLE001 (handed to the test)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    t = time.perf_counter()
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    return time.perf_counter() - t, out


@pytest.mark.parametrize("s,n,k,count", [(64_000, 16, 25, 12), (20_000, 64, 40, 5), (700, 3, 6, 40)])
def test_results_do_not_depend_on_other_calls(s, n, k, count):
    jobs = _jobs(s, n, k, count)
    kpp, ll = [_kpp(j) for j in jobs], [_lloyd(j) for j in jobs]
    for a, b in zip(_together(_kpp, jobs, 3)[1], kpp):
        assert torch.equal(a, b)
    for a, b in zip(_together(_lloyd, jobs, 3)[1], ll):
        assert torch.equal(a[0], b[0]) and a[1:3] == b[1:3] and torch.equal(a[3], b[3])


def test_eight_threads_seed_at_least_twice_as_fast_as_one():
    jobs = _jobs(64_000, 16, 25, 8)
    _together(_kpp, jobs, 2)
    best = 0.0
    for _ in range(4):
        one = _together(_kpp, jobs[:1], 24)[0] / 24
        best = max(best, one / (_together(_kpp, jobs, 24)[0] / (8 * 24)))
    assert best >= 2.0, best

"""Greedy K-means++ at the sizes where its one-exchange form can go wrong: fewer rows than warps,
rows at the edges of warps and CTAs, every padded width (the distances are cut short in chunks of
dimensions), a largest D^2 whose exponent falls at every pick (the quantisation grid changes), one
to three candidates, and groups of clusters.  All results are integers or rows of the sample:
bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import bigmeans as obm
from oracle import kmeans as okm
from oracle import rng as orng
from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture

pytestmark = pytest.mark.gpu


def _check(S, k, trials, seed, deg=None, C0=None):
    deg = np.ones(k, bool) if deg is None else deg
    C0 = np.zeros((k, S.shape[1]), np.float32) if C0 is None else C0
    got = native.kmeanspp(torch.from_numpy(S).cuda(), torch.from_numpy(C0).cuda(), deg.astype(np.uint8), trials, seed,
                          1, 2, 3).cpu().numpy()
    ref, _ = okm.kmeanspp_reseed(S, C0, deg, orng.stream_key(seed, orng.P_KPP, 1, 2, 3), trials)
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("s,k", [(2, 2), (5, 5), (31, 9), (255, 12), (257, 12), (1025, 20), (4100, 33)])
@pytest.mark.parametrize("n", [1, 7, 12, 30, 50])
@pytest.mark.parametrize("trials", [1, 2, 3])
def test_edges_of_warps_and_ctas(s, k, n, trials):
    _check(gaussian_mixture(s, n, max(1, k // 2), seed=s + n), k, trials, seed=s)


@pytest.mark.parametrize("n", [2, 16, 32, 64])
def test_falling_exponent_of_the_largest_distance(n):
    rng = np.random.default_rng(n)
    S = (rng.standard_normal((3000, n)) * np.exp2(rng.uniform(-30, 10, (3000, 1)))).astype(np.float32)
    _check(S, 40, 3, seed=5)
    deg = np.arange(40) % 3 == 1
    _check(S, 40, 3, seed=6, deg=deg, C0=S[:40].copy())


def test_more_centroids_than_distinct_rows():
    S = np.repeat(np.random.default_rng(1).standard_normal((6, 20)).astype(np.float32), 50, axis=0)
    _check(S, 9, 3, seed=7)


@pytest.mark.parametrize("n,k,s_max", [(64, 40, 9000), (16, 25, 30000), (3, 6, 2500)])
def test_groups_of_clusters(n, k, s_max):
    """Two workers share the device: each spans several clusters, which all take part in the seeding."""
    X = gaussian_mixture(40_000, n, k, seed=n)
    pol = dict(s_min=s_max // 2, s_max=s_max, workers=2, passes=2)
    bud = dict(rounds=1, max_lloyd=20, tol=1e-4, kpp_candidates=3)
    ref = obm.bigmeans(X, k, pol, bud, seed=9)
    outs = []
    try:
        for on in (1, 0):
            native.set_worker_groups(on)
            outs.append(native.fit(torch.from_numpy(X).cuda(), k, native.make_policy(**pol),
                                   native.make_budget(**bud), seed=9))
    finally:
        native.set_worker_groups(1)
    for C, Y, rep in outs:
        assert np.array_equal(C.cpu().numpy().view(np.uint32), ref["C"].view(np.uint32))
        assert np.array_equal(Y.cpu().numpy(), ref["labels"]) and rep["f_full"] == ref["f_full"]

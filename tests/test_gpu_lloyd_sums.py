"""The exact sums of a Lloyd run where their forms meet: coordinates above and below the unit that one
64-bit half holds (2^-24 of the largest |x|) in the same batch and cluster, clusters of a few rows
beside very large ones (bucket boundaries inside a warp's share of the rows), more than 32 clusters,
every padded width, and more rows per thread than the 64-bit objective sums take before they are
folded into 128 bits.  C and f equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

from oracle import kmeans as okm
from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture

pytestmark = pytest.mark.gpu


def _check(S, C0, max_iter=6, tol=0.0):
    C, f, it, empty = native.lloyd(torch.from_numpy(S).cuda(), torch.from_numpy(C0).cuda(), max_iter, tol)
    ref = okm.lloyd(S, C0, max_iter, tol)
    assert it == ref["iters"] and f == ref["f"]
    assert np.array_equal(C.cpu().numpy().view(np.uint32), ref["C"].view(np.uint32))
    assert np.array_equal(empty.cpu().numpy(), ref["empty"])


@pytest.mark.parametrize("n", [1, 4, 7, 16, 23, 64])
@pytest.mark.parametrize("k", [2, 33, 70])
def test_mixed_magnitudes_and_cluster_sizes(n, k):
    rng = np.random.default_rng(100 * n + k)
    s = 3000
    # most rows in two clusters, the others in clusters of one to three rows, in random order
    sizes = [1 + j % 3 for j in range(k - 2)]
    sizes = [(s - sum(sizes)) // 2] * 2 + sizes
    sizes[0] += s - sum(sizes)
    cent = (rng.standard_normal((k, n)) * 8).astype(np.float32)
    lab = rng.permutation(np.repeat(np.arange(k), sizes))
    S = (cent[lab] + rng.standard_normal((s, n)) * 0.01).astype(np.float32)
    # a third of the coordinates 2^-1 to 2^-60 of the others: whole batches of them, and mixed ones
    small = rng.random((s, n)) < np.where(lab % 2, 0.05, 0.6)[:, None]
    S = np.where(small, S * np.exp2(rng.uniform(-60, -1, (s, n))), S).astype(np.float32)
    S[rng.integers(0, s, 20)] = 0
    _check(S, cent)


@pytest.mark.parametrize("scale", [1e-36, 1e-20, 1e18])
def test_mixed_magnitudes_near_the_ends_of_the_range(scale):
    rng = np.random.default_rng(5)
    S = (rng.standard_normal((2000, 12)) * np.exp2(rng.uniform(-40, 0, (2000, 12))) * scale).astype(np.float32)
    _check(S, S[:40].copy())


@pytest.mark.parametrize("n", [2, 5])
def test_more_than_64_rows_per_thread(n):
    S = gaussian_mixture(300_000, n, 4, seed=n)
    try:
        native.set_worker_groups(0)              # one cluster of 16 CTAs: 18,750 rows each
        _check(S, S[:4].copy(), max_iter=2)
    finally:
        native.set_worker_groups(1)

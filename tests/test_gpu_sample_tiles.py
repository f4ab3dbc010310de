"""Samples lie in tiles of four rows and a warp's trip takes as many rows per lane as leaves no warp
idle: gather, Lloyd and seeding at row counts around the tile, the warp and the trip, at every
padded width, against the oracle (bit-exact)."""
import numpy as np
import pytest
import torch

from oracle import kmeans as okm
from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 6, 9, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("s", [1, 3, 4, 5, 33, 258])
def test_gather_round_trip(n, s):
    X = np.random.default_rng(s * n).standard_normal((300, n)).astype(np.float32)
    idx = np.random.default_rng(s).permutation(300)[:s].astype(np.int64)
    S = native.gather(torch.from_numpy(X).cuda(), torch.from_numpy(idx).cuda()).cpu().numpy()
    assert np.array_equal(S, X[idx])


@pytest.mark.parametrize("n,k", [(2, 4), (8, 5), (13, 6), (20, 9), (64, 7)])
@pytest.mark.parametrize("s", [9, 31, 255, 256, 257, 513, 1023, 2049, 2300])
def test_lloyd_row_counts(n, k, s):
    S = gaussian_mixture(s, n, k, seed=s + n)
    C0 = S[np.linspace(0, s - 1, k).astype(int)].copy()
    C, f, it, empty = native.lloyd(torch.from_numpy(S).cuda(), torch.from_numpy(C0).cuda(), 10, 1e-4)
    ref = okm.lloyd(S, C0, 10, 1e-4)
    assert np.array_equal(C.cpu().numpy().view(np.uint32), ref["C"].view(np.uint32))
    assert f == ref["f"] and it == ref["iters"]


@pytest.mark.parametrize("n,k,s", [(2, 5, 100_003), (16, 25, 70_001), (32, 50, 131_072), (64, 20, 40_000)])
def test_step_calls_on_a_group_of_clusters(n, k, s):
    """One worker on many clusters (the group's sums are added in three buffers in turn, so more than
    three Lloyd exchanges) gives the bits of one cluster."""
    S = torch.from_numpy(gaussian_mixture(s, n, k, seed=n + k)).cuda()
    C0 = S[torch.linspace(0, s - 1, k).long().cuda()].clone()
    outs = []
    try:
        for on in (1, 0):
            native.set_worker_groups(on)
            C, f, it, empty = native.lloyd(S, C0, 12, 0.0)
            P = native.kmeanspp(S, C0, np.arange(k) % 2, 3, 5, 0, 0, 0)
            outs.append((C, f, it, empty, P))
    finally:
        native.set_worker_groups(1)
    a, b = outs
    assert a[2] == b[2] >= 4 and a[1] == b[1] and torch.equal(a[3], b[3])
    assert torch.equal(a[0].view(torch.int32), b[0].view(torch.int32))
    assert torch.equal(a[4].view(torch.int32), b[4].view(torch.int32))

"""The tensor-core full pass on rows whose magnitudes span several decades: the certificate of a row
depends on its own norm and its own distance, so that a few far centroids don't make all rows keep
many candidates.  Labels and f equal the FP32-ALU pass bit for bit."""
import pytest
import torch

from paper_2403_18766_gb300 import native

pytestmark = pytest.mark.gpu

M = 131_073


def _rows(n, sigma, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.exp(sigma * torch.randn((M, n), generator=g, device="cuda"))


def _tensor_and_alu(X, C):
    try:
        native.set_fullpass_impl(0)
        Y0, f0, r0 = native.assign(X, C)
        assert native.last_fullpass_impl() == 2
        native.set_fullpass_impl(1)
        Y1, f1, r1 = native.assign(X, C)
    finally:
        native.set_fullpass_impl(0)
    assert torch.equal(Y0, Y1) and f0 == f1 and r0["inexact_terms"] == r1["inexact_terms"]
    return r0["rescored_rows"]


@pytest.mark.parametrize("n,k", [(4, 200), (8, 60), (12, 25), (13, 100), (16, 200), (21, 33), (32, 50), (61, 90),
                                 (64, 256)])
@pytest.mark.parametrize("sigma", [1.0, 3.0, 6.0])
def test_log_normal_rows(n, k, sigma):
    X = _rows(n, sigma, seed=n + k)
    _tensor_and_alu(X, X[torch.linspace(0, M - 1, k).long().cuda()].clone())


@pytest.mark.parametrize("n", [8, 16, 40])
def test_a_far_centroid_leaves_the_other_rows_as_they_are(n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    X = torch.randn((M, n), generator=g, device="cuda")
    C = X[:63].clone()
    base = _tensor_and_alu(X, C)
    C[17] = 1e4
    assert _tensor_and_alu(X, C) <= 2 * base + M // 100

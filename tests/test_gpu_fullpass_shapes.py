"""The tensor-core full pass at the edges of its forms: one, four and eight mask words, centroids in
shared and in global memory, widths that are no multiple of 4 (contiguous copies, also with a last
tile whose bytes are no multiple of 16), an odd stage count, ties across mask words, magnitudes near
the FP32 range and near zero.  Labels and f equal the FP32-ALU pass, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture_device

pytestmark = pytest.mark.gpu

M = 131_073                      # from here the default takes the tensor cores for every width


def _same(X, C, want_tensor=True):
    try:
        native.set_fullpass_impl(0)
        Y0, f0, r0 = native.assign(X, C)
        i0 = native.last_fullpass_impl()
        native.set_fullpass_impl(1)
        Y1, f1, r1 = native.assign(X, C)
    finally:
        native.set_fullpass_impl(0)
    assert i0 == (2 if want_tensor else 1)
    assert torch.equal(Y0, Y1) and f0 == f1 and r0["inexact_terms"] == r1["inexact_terms"]


@pytest.mark.parametrize("n,k", [(4, 64), (7, 97), (8, 32), (8, 33), (13, 48), (16, 16), (16, 128), (16, 129),
                                 (21, 33), (30, 256), (32, 8), (32, 100), (32, 256), (35, 12), (36, 31), (63, 12),
                                 (63, 160), (64, 4), (64, 32), (64, 33), (64, 128), (64, 129), (64, 256)])
@pytest.mark.parametrize("m", [M, M + 126])
def test_forms_of_the_pass(m, n, k):
    X = gaussian_mixture_device(m, n, max(1, k // 2), seed=n * k + m)
    _same(X, X[torch.linspace(0, m - 1, k).long().cuda()].clone())


@pytest.mark.parametrize("n,k", [(16, 200), (21, 90), (64, 70)])
def test_ties_across_mask_words(n, k):
    X = gaussian_mixture_device(M, n, 5, seed=3)
    C = X[:k].clone()
    C[k - 1] = C[0]
    C[k // 2] = C[0]
    C[40:50] = C[1]
    _same(X, C)


@pytest.mark.parametrize("scale", [1e-30, 1e-18, 1e15, 1e18, 3e37])
@pytest.mark.parametrize("n", [8, 17, 64])
def test_magnitudes(n, scale):
    X = gaussian_mixture_device(M, n, 8, seed=4) / 16 * scale
    _same(X, X[:48].clone())


def test_rows_far_from_the_centroids_and_zero_rows():
    X = gaussian_mixture_device(M, 32, 8, seed=5)
    X[::7] *= 1e6
    X[::11] = 0
    _same(X, X[1:40].clone())


@pytest.mark.parametrize("m,n,k,tensor", [(131_072, 16, 25, False), (M, 16, 25, True), (M, 16, 15, False),
                                          (M, 21, 23, False), (M, 21, 24, True), (131_072, 21, 200, False)])
def test_choice_by_rows(m, n, k, tensor):
    X = gaussian_mixture_device(m, n, 6, seed=6)
    _same(X, X[:k].clone(), tensor)


@pytest.mark.parametrize("k", [1, 5, 16, 17, 20, 31, 32, 33, 47, 49, 64, 97, 100, 129, 256])
def test_precision_form_column_edges(k):
    """The candidate masks of the BF16 pass at the edges of its chunks of 16 and 32 columns: the
    certified form's labels are the exact pass's, and tau = inf gives its f too."""
    X = gaussian_mixture_device(20_000, 50, max(1, k // 2), seed=k)
    C = X[torch.linspace(0, 19_999, k).long().cuda()].clone()
    P = native.PackedBF16(X)
    Y, f, _ = native.assign(X, C)
    assert torch.equal(native.assign_bf16(P, C, tau=0.0, certified=True)[0], Y)
    Yi, fi, _ = native.assign_bf16(P, C, tau=float("inf"))
    assert torch.equal(Yi, Y) and fi == f

"""The tensor-core full pass on rows far from the origin: its operands are shifted by a mean of
centroids, so that the rows' common offset leaves the certificate as it is.  Labels and f equal the
FP32-ALU pass bit for bit, and about as many rows have several candidates as without the offset."""
import pytest
import torch

from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture_device

pytestmark = pytest.mark.gpu

M = 131_073 + 4000               # tensor cores for every width, a ragged last tile


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


# four and eight mask words (k > 32: where rows are shifted), every padded width, contiguous copies,
# centroids in global memory
@pytest.mark.parametrize("n,k", [(4, 130), (8, 100), (16, 33), (16, 200), (21, 33), (32, 50), (61, 90), (64, 100),
                                 (64, 256)])
@pytest.mark.parametrize("offset", [300.0, -3000.0])
def test_an_offset_leaves_few_rows_with_several_candidates(n, k, offset):
    X = gaussian_mixture_device(M, n, k, seed=n + k)
    C = X[torch.linspace(0, M - 1, k).long().cuda()].clone()
    base = _tensor_and_alu(X, C)
    u = offset * torch.linspace(0.5, 1.0, n, device="cuda")
    # the rows keep 24 bits, so an offset of 3000 blurs them by 2^-13 and moves a few
    assert _tensor_and_alu(X + u, C + u) <= 2 * base + M // 50


@pytest.mark.parametrize("n", [8, 33, 64])
@pytest.mark.parametrize("offset", [1e-32, 1e6, 2.0 ** 100, 1.5 * 2.0 ** 125])
def test_offsets_of_all_magnitudes(n, offset):
    """Also where the offset swallows the rows' differences, and where sums of rows leave FP32."""
    X = gaussian_mixture_device(M, n, 8, seed=n) * (abs(offset) / 64 if offset < 1 else 1.0) + offset
    _tensor_and_alu(X, X[:96].clone())


@pytest.mark.parametrize("k", [17, 48, 140])
def test_groups_of_opposite_sign_and_one_far_centroid(k):
    X = gaussian_mixture_device(M, 24, 6, seed=k)
    X[::2] += 500.0
    X[1::2] -= 400.0
    C = X[:k].clone()
    _tensor_and_alu(X, C)
    C[0] = 1e9
    _tensor_and_alu(X, C)


def test_one_centroid():
    X = gaussian_mixture_device(M, 64, 3, seed=1) + 77.0
    try:
        native.set_fullpass_impl(2)
        Y, f, r = native.assign(X, X[:1].clone())
        native.set_fullpass_impl(1)
        Y1, f1, _ = native.assign(X, X[:1].clone())
    finally:
        native.set_fullpass_impl(0)
    assert torch.equal(Y, Y1) and f == f1 and r["rescored_rows"] == 0

"""The contiguous-copy form of the tensor-core full pass (n % 4 != 0) at its smallest pieces: a last
tile of one row whose bytes are no multiple of 16 (none, for n < 4), and bounded waits that run out."""
import pytest
import torch

from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture_device

pytestmark = pytest.mark.gpu


def _both(X, C):
    try:
        native.set_fullpass_impl(0)
        Y0, f0, _ = native.assign(X, C)
        impl = native.last_fullpass_impl()
        native.set_fullpass_impl(1)
        Y1, f1, _ = native.assign(X, C)
    finally:
        native.set_fullpass_impl(0)
    assert torch.equal(Y0, Y1) and f0 == f1
    return impl


@pytest.mark.parametrize("n,k", [(2, 192), (3, 200), (5, 100), (9, 60), (33, 40)])
@pytest.mark.parametrize("m", [131_073, 131_074, 131_199, 131_200])
def test_last_tiles(m, n, k):
    X = gaussian_mixture_device(m, n, 7, seed=m + n)
    assert _both(X, X[torch.linspace(0, m - 1, k).long().cuda()].clone()) == 2


def test_one_column_takes_the_alu_pass():
    X = gaussian_mixture_device(131_073, 1, 7, seed=5)
    assert _both(X, X[:200].clone()) == 1


def test_wait_that_runs_out():
    X = gaussian_mixture_device(140_001, 21, 9, seed=3)
    C = X[:40].clone()
    Y, f, _ = native.assign(X, C)
    assert native.last_fullpass_impl() == 2
    timeouts = 0
    try:
        native.debug_set_wait_limit(1, 0)          # one plain poll per wait
        for _ in range(4):
            try:
                Y1, f1, _ = native.assign(X, C)
            except native.BigmeansError as e:
                assert e.status == native.BM_ETIMEOUT, str(e)
                timeouts += 1
                continue
            assert torch.equal(Y, Y1) and f == f1  # a call that did not run out
    finally:
        native.debug_set_wait_limit(0)
    assert timeouts >= 1
    Y1, f1, _ = native.assign(X, C)
    assert torch.equal(Y, Y1) and f == f1

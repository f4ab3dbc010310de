"""The input scan and the BF16 pack at their edges: unaligned pointers, row counts around the
tile of 128, widths with and without 16-byte rows, non-finite values at either end."""
import numpy as np
import pytest
import torch

from paper_2403_18766_gb300 import native

pytestmark = pytest.mark.gpu


def _bf16(x):
    """Round to nearest even to 8 significant bits (finite values)."""
    b = x.view(np.uint32).astype(np.uint64)
    return (((b + 0x7fff + ((b >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("m", [1, 127, 128, 129, 1000])
@pytest.mark.parametrize("n", [1, 3, 4, 20, 31, 61, 64])
@pytest.mark.parametrize("shift", [0, 1])
def test_pack_layout_norms_and_max(m, n, shift):
    rng = np.random.default_rng(m * 100 + n)
    x = (rng.standard_normal((m, n)) * 10).astype(np.float32)
    raw = torch.zeros(m * n + 4, device="cuda")
    X = raw[shift:shift + m * n].view(m, n)             # shift 1: rows off the 16-byte grid
    X.copy_(torch.from_numpy(x))
    P = native.PackedBF16(X)
    m_pad = (m + 127) // 128 * 128
    want = np.zeros((m_pad, 64), np.float32)
    want[:m, :n] = _bf16(x)
    got = P.Xb.cpu().numpy().view(np.uint16).reshape(m_pad, 8, 8)
    r = np.arange(m_pad)[:, None]
    got = got[r, np.arange(8)[None, :] ^ (r & 7)].reshape(m_pad, 64)
    assert np.array_equal(got, (want.view(np.uint32) >> 16).astype(np.uint16))
    norms = P.norms.cpu().numpy()
    # an FMA chain: each partial sum is the exact sum rounded once (64-bit products of 8-bit
    # significands are exact, the 64-bit sum of two floats is exact to far below a half ulp here)
    acc = np.zeros(m_pad, np.float32)
    for d in range(64):
        acc = (acc.astype(np.float64) + want[:, d].astype(np.float64) ** 2).astype(np.float32)
    assert np.array_equal(norms[:m_pad], acc)
    assert norms[m_pad] == np.abs(x).max()


@pytest.mark.parametrize("m,n", [(1, 1), (5, 3), (4097, 4), (70001, 5)])
@pytest.mark.parametrize("where", ["first", "last", "middle"])
@pytest.mark.parametrize("bad", [float("nan"), float("-inf")])
def test_scan_finds_non_finite_values(m, n, where, bad):
    X = torch.ones((m, n), device="cuda")
    flat = X.view(-1)
    flat[{"first": 0, "last": m * n - 1, "middle": m * n // 2}[where]] = bad
    with pytest.raises(native.BigmeansError, match="1 non-finite"):
        native.assign(X, torch.zeros((1, n), device="cuda"))
    C = torch.full((1, n), bad, device="cuda")
    with pytest.raises(native.BigmeansError, match=f"{n} non-finite"):
        native.assign(torch.ones((m, n), device="cuda"), C)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("s", [1, 2, 3, 6, 1025])
def test_scan_of_an_unaligned_sample(s, shift):
    """bm_lloyd takes a sample at any 4-byte address; the largest value decides the grid of the
    exact sums, wherever it lies, so the result equals the aligned one's."""
    n = 3
    g = np.random.default_rng(s + shift)
    x = g.standard_normal((s, n)).astype(np.float32)
    x[-1, -1] = 1e20
    raw = torch.zeros(s * n + 4, device="cuda")
    A = raw[shift:shift + s * n].view(s, n)
    A.copy_(torch.from_numpy(x))
    C = torch.from_numpy(x[:1].copy()).cuda()
    a = native.lloyd(A, C, max_iter=3)
    b = native.lloyd(torch.from_numpy(x).cuda(), C, max_iter=3)
    assert torch.equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2]
    assert np.isfinite(a[1])


@pytest.mark.parametrize("n", [31, 61])
def test_pack_of_odd_widths_keeps_up_with_even_ones(n):
    """Rows that are no multiple of 16 bytes take at most half as long again as those one wider."""
    def us(X):
        for _ in range(3):
            native.PackedBF16(X)
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            native.PackedBF16(X)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        return best

    m = 4_000_000
    assert us(torch.randn((m, n), device="cuda")) <= 1.5 * us(torch.randn((m, n + 1), device="cuda"))

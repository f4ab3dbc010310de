"""Samples drawn by many CTAs per job equal the oracle's (the first s distinct draws, in order):
sizes around the chunk of 1024 draws and the switch-over, few and many repeats (s up to m / 2), jobs
of very different sizes in one launch, step calls, fits, and fits that change between the samplers."""
import numpy as np
import pytest
import torch

from oracle import bigmeans as obm
from oracle import rng as orng
from paper_2403_18766_gb300 import native
from paper_2403_18766_gb300.synthetic import gaussian_mixture

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,s", [(8192, 4096), (8191, 4095), (10_001, 5000), (100_000, 4096), (100_003, 50_001),
                                 (4_000_000, 4097), (4_000_000, 131_072), (2_000_000_000, 70_001),
                                 (1_048_544, 524_272)])
def test_samples_equal_the_oracle_and_the_tables(m, s):
    got = native.sample(11, native.RNG_PASS, 3, 4, 5, m, s).cpu().numpy()
    try:
        native.set_sampler_impl(1)
        tab = native.sample(11, native.RNG_PASS, 3, 4, 5, m, s).cpu().numpy()
    finally:
        native.set_sampler_impl(0)
    assert np.array_equal(got, tab)
    assert len(np.unique(got)) == s and got.min() >= 0 and got.max() < m
    if s <= 131_072:
        assert np.array_equal(got, obm.sample_indices(11, orng.P_PASS, 3, 4, 5, m, s))


@pytest.mark.parametrize("n", [3, 8, 20, 64])
def test_fit_equals_the_oracle(n):
    X = gaussian_mixture(30_000, n, 5, seed=n)
    pol = dict(s_min=300, s_max=6000, workers=3, passes=2)
    bud = dict(rounds=3, max_lloyd=20, tol=1e-4, kpp_candidates=3)
    C, Y, rep = native.fit(torch.from_numpy(X).cuda(), 5, native.make_policy(**pol), native.make_budget(**bud), seed=3)
    ref = obm.bigmeans(X, 5, pol, bud, seed=3)
    assert np.array_equal(C.cpu().numpy().view(np.uint32), ref["C"].view(np.uint32))
    assert np.array_equal(Y.cpu().numpy(), ref["labels"]) and rep["f_full"] == ref["f_full"]
    assert rep["s_opt"] == ref["s_opt"]


def test_changing_the_sampler_between_rounds():
    X = torch.from_numpy(gaussian_mixture(60_000, 8, 5, seed=2)).cuda()
    pol, bud = native.make_policy(s_min=500, s_max=9000, workers=3, passes=2), native.make_budget(rounds=6)
    C0, Y0, r0 = native.fit(X, 5, pol, bud, seed=4)
    sess = native.FitSession(X, 5, pol, bud, seed=4)
    try:
        for r in range(6):
            native.set_sampler_impl(r // 2 % 2)
            sess.rounds(1)
        C1, Y1, r1 = sess.finish()
    finally:
        native.set_sampler_impl(0)
        sess.close()
    assert torch.equal(C0.view(torch.int32), C1.view(torch.int32)) and torch.equal(Y0, Y1)
    assert r0["f_full"] == r1["f_full"]


@pytest.mark.parametrize("n", [1, 4, 7, 64])
def test_gather_checks_every_index(n):
    X = torch.randn((500, n), device="cuda")
    idx = torch.randint(0, 500, (3000,), device="cuda")
    assert torch.equal(native.gather(X, idx), X[idx])
    for bad in (-1, 500):
        idx[1234] = bad
        with pytest.raises(native.BigmeansError) as e:
            native.gather(X, idx)
        assert e.value.status == native.BM_EINVAL


@pytest.mark.parametrize("rounds", [1, 3])
def test_every_kernel_of_a_sampling_launch_is_counted(rounds):
    """Three kernels per launch with many CTAs per job (here the first round's and the final sample;
    the rounds drawn ahead take one), one with a CTA per job."""
    X = torch.from_numpy(gaussian_mixture(60_000, 8, 5, seed=2)).cuda()
    pol, bud = native.make_policy(s_min=500, s_max=9000, workers=3, passes=2), native.make_budget(rounds=rounds)
    counts = []
    try:
        for impl in (0, 1):
            native.set_sampler_impl(impl)
            counts.append(native.fit(X, 5, pol, bud, seed=4)[2]["kernel_launches"])
    finally:
        native.set_sampler_impl(0)
    assert counts[0] == counts[1] + 4


def test_generations_start_again():
    """A fit of more rounds than a table slot has generations clears both halves of its tables and goes
    on: every sample is drawn by many CTAs (2 10^6 rows are too many for the bitmap), and the result
    is that of one CTA per sample."""
    rounds = 8300
    X = torch.from_numpy(gaussian_mixture(40_000, 1, 4, seed=3)).cuda().repeat(50, 1).contiguous()
    pol = native.make_policy(s_min=4100, s_max=4200, workers=1, passes=1)
    bud = native.make_budget(rounds=rounds, max_lloyd=1)
    outs = []
    try:
        for impl in (0, 1):
            native.set_sampler_impl(impl)
            outs.append(native.fit(X, 2, pol, bud, seed=8))
    finally:
        native.set_sampler_impl(0)
    (C0, Y0, r0), (C1, Y1, r1) = outs
    assert r0["rounds_done"] == rounds and r0["kernel_launches"] >= 4 * rounds
    assert torch.equal(C0, C1) and torch.equal(Y0, Y1) and r0["f_full"] == r1["f_full"]
    assert r0["accepts"] == r1["accepts"] and r0["L_sum"] == r1["L_sum"]

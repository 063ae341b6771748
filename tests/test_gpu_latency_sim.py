"""The CUDA latency simulations against the CPU oracle, trial by trial (same
counter-based random stream on both sides, float64; the only differences are
last-digit roundings of log/cos/exp), plus the closed forms at any size."""

import math

import numpy as np
import pytest

from oracle import latency_oracle as L

pytestmark = pytest.mark.gpu
RTOL = 1e-11


@pytest.fixture(scope="module")
def nolo():
    from paper_2506_10911_b200 import binding
    return binding


@pytest.mark.parametrize("W,mu,sigma,trials,seed", [
    (2, 0.5, 0.8, 50, 3), (4, 0.0, 1.0, 40, 2), (64, 1.0, math.sqrt(0.5), 12, 9), (1024, -0.3, 0.25, 3, 1),
    (4096, 0.0, 0.5, 1, 5), (8, 0.0, 1.0, 300, 4), (32, 0.2, 0.7, 70, 4), (128, 0.2, 0.7, 5, 4), (512, 0.1, 1.0, 2, 4),
])
def test_tree_allreduce_trials_match_oracle(nolo, W, mu, sigma, trials, seed):
    mean, se, per = nolo.nolo_sim_tree_allreduce(W, mu, sigma, trials, seed, return_trials=True)
    want = L.sim_tree_allreduce(W, mu, sigma, trials, seed)
    np.testing.assert_allclose(per, want, rtol=RTOL)
    assert mean == pytest.approx(want.mean(), rel=RTOL)
    if trials > 1:
        assert se == pytest.approx(want.std(ddof=1) / math.sqrt(trials), rel=1e-9)


def test_tree_allreduce_closed_forms_at_scale(nolo):
    for W in (2, 32, 1024):
        mean, se = nolo.nolo_sim_tree_allreduce(W, 0.3, 0.0, 100, 1)
        assert mean == pytest.approx(2 * math.exp(0.3) * math.log2(W), rel=1e-13) and se < 1e-12
    mu, sigma = 0.5, 0.8
    mean, se = nolo.nolo_sim_tree_allreduce(2, mu, sigma, 400_000, 7)
    closed = nolo.nolo_expected_pair_exchange(mu, sigma)
    assert closed == pytest.approx(L.expected_pair_exchange(mu, sigma), rel=1e-15)
    assert abs(mean - closed) < 4.5 * se                       # the appendix's E[max] formula
    # Fig. 5a: the advantage over pair exchange grows with W and with the variance
    r = {(W, s): nolo.nolo_sim_tree_allreduce(W, 0.0, s, 20_000, 11)[0] / nolo.nolo_expected_pair_exchange(0.0, s)
         for W in (4, 64, 1024) for s in (0.1, 1.0)}
    assert r[(4, 1.0)] < r[(64, 1.0)] < r[(1024, 1.0)]
    assert r[(1024, 1.0)] > r[(1024, 0.1)] > 0.99 * 10


@pytest.mark.parametrize("W,n,H,T,trials,seed", [
    (4, 2, 3, 2, 5, 11), (16, 4, 10, 6, 4, 2), (8, 8, 5, 7, 3, 4), (1, 1, 4, 3, 2, 0), (100, 5, 7, 4, 2, 6),
    (1024, 2, 100, 4, 1, 0), (2048, 2, 3, 2, 1, 8),
])
def test_straggler_trials_match_oracle(nolo, W, n, H, T, trials, seed):
    mu, sigma = 1.0, math.sqrt(0.5)
    *stats, per = nolo.nolo_sim_straggler(W, n, H, T, mu, sigma, trials, seed, return_trials=True)
    want = L.sim_straggler(W, n, H, T, mu, sigma, trials, seed)
    np.testing.assert_allclose(per, want, rtol=RTOL)
    assert stats[0] == pytest.approx(want[:, 0].mean(), rel=RTOL)
    assert stats[1] == pytest.approx(want[:, 1].mean(), rel=RTOL)
    assert (per[:, 1] <= per[:, 0] * (1 + 1e-15)).all()


@pytest.mark.parametrize("W,n,H,T,trials", [
    (2, 1, 1, 1, 3), (31, 31, 5, 3, 2), (32, 16, 4, 3, 2), (33, 11, 9, 3, 2), (96, 48, 33, 2, 2), (512, 128, 3, 2, 1),
    (513, 27, 3, 2, 1), (1025, 205, 3, 2, 1), (4096, 4096, 2, 2, 1), (4096, 1, 130, 1, 1),
])
def test_straggler_kernel_boundaries(nolo, W, n, H, T, trials):
    """Sizes where the kernels change: warps or CTAs of 128, 512 or 1024 threads per partition, subgroups
    shared by up to 32 threads, items shared by up to 32 threads, inner steps that fill no block."""
    *_, per = nolo.nolo_sim_straggler(W, n, H, T, 0.5, 0.9, trials, 12, return_trials=True)
    np.testing.assert_allclose(per, L.sim_straggler(W, n, H, T, 0.5, 0.9, trials, 12), rtol=RTOL)


@pytest.mark.parametrize("trials", [1, 2, 4095, 8191, 8192, 8193, 12_289, 300_001])
def test_means_and_standard_errors_of_many_trials(nolo, trials):
    """The rows are summed in slices of 4096 and more, 64 at most; float64 sums of up to 3e5 terms of one sign."""
    mean, se, per = nolo.nolo_sim_tree_allreduce(2, 0.1, 0.6, trials, 5, return_trials=True)
    assert mean == pytest.approx(per.mean(), rel=1e-13)
    assert se == (pytest.approx(per.std(ddof=1) / math.sqrt(trials), rel=1e-11) if trials > 1 else 0.0)
    b, s, eb, es, per = nolo.nolo_sim_straggler(2, 1, 1, 1, 0.1, 0.6, trials, 5, return_trials=True)
    assert (b, s) == pytest.approx(tuple(per.mean(0)), rel=1e-13)
    if trials > 1:
        assert (eb, es) == pytest.approx(tuple(per.std(0, ddof=1) / math.sqrt(trials)), rel=1e-11)


def test_straggler_in_slabs_agrees_with_itself(nolo):
    """2^21 work sums are held at a time.  The first trials of a call that needs several slabs of
    iterations (and of trials) have the times that a call of those trials alone gives."""
    for W, T, trials in ((2048, 30, 40), (4096, 3, 600)):
        *_, per = nolo.nolo_sim_straggler(W, 2, 2, T, 0.0, 0.5, trials, 3, return_trials=True)
        *_, few = nolo.nolo_sim_straggler(W, 2, 2, T, 0.0, 0.5, 2, 3, return_trials=True)
        np.testing.assert_allclose(per[:2], few, rtol=1e-14)
        assert (per[:, 1] <= per[:, 0] * (1 + 1e-15)).all() and (per > 0).all()


@pytest.mark.parametrize("mu,sigma", [(0.0, 80.0), (690.0, 0.5), (705.0, 1.0), (-740.0, 0.1), (0.0, 0.0), (0.0, 400.0)])
def test_times_at_the_ends_of_the_range(nolo, mu, sigma):
    """Times that leave the normal numbers are taken by the general form of exp; either form agrees with
    the oracle (relative to e^|exponent|'s own rounding: 2^-53 of an exponent of 700 is 8e-14)."""
    with np.errstate(over="ignore"):
        want = L.sim_tree_allreduce(16, mu, sigma, 40, 8)
    *_, per = nolo.nolo_sim_tree_allreduce(16, mu, sigma, 40, 8, return_trials=True)
    np.testing.assert_allclose(per, want, rtol=1e-11, atol=1e-320)


def test_straggler_reproduces_the_papers_figure_at_full_size(nolo):
    """W = 1024, pairs, 100 inner steps per outer step, 250 outer iterations,
    LogNormal(1, 0.5): the global barrier costs about 20 % (Section 4.3)."""
    b, s, eb, es = nolo.nolo_sim_straggler(1024, 2, 100, 250, 1.0, math.sqrt(0.5), 8, 0)
    assert 1.14 < b / s < 1.26
    # no variance -> nobody waits
    b, s, _, _ = nolo.nolo_sim_straggler(1024, 2, 100, 5, 1.0, 0.0, 2, 0)
    assert b == pytest.approx(500 * math.e, rel=1e-12) and s == pytest.approx(b, rel=1e-15)


def test_simulations_from_several_threads_and_streams(nolo):
    """Each call has scratch of its own: calls that overlap give what they give alone, also when handles
    are destroyed in between (which gives kept scratch back)."""
    import threading
    import torch
    want = {s: (nolo.nolo_sim_tree_allreduce(64, 0.0, 1.0, 5000, s, return_trials=True)[2],
                nolo.nolo_sim_straggler(64, 2, 10, 20, 0.0, 0.5, 40, s, return_trials=True)[4]) for s in range(6)}
    bad = []

    def work(s):
        stream = torch.cuda.Stream()
        for _ in range(10):
            a = nolo.nolo_sim_tree_allreduce(64, 0.0, 1.0, 5000, s, stream, return_trials=True)[2]
            b = nolo.nolo_sim_straggler(64, 2, 10, 20, 0.0, 0.5, 40, s, stream, return_trials=True)[4]
            nolo.nolo_destroy(nolo.nolo_create(2, 1, 8, 1, 0.5, 0.7, 0.5))
            if not (np.array_equal(a, want[s][0]) and np.array_equal(b, want[s][1])):
                bad.append(s)

    threads = [threading.Thread(target=work, args=(s,)) for s in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_simulation_argument_checks(nolo):
    for bad in [(6, 0.0, 1.0, 10), (1, 0.0, 1.0, 10), (8, 0.0, -1.0, 10), (8, 0.0, 1.0, 0), (8, float("nan"), 1.0, 1)]:
        with pytest.raises(nolo.NoloError) as e:
            nolo.nolo_sim_tree_allreduce(bad[0], bad[1], bad[2], bad[3], 0)
        assert e.value.status == nolo.NOLO_EINVAL
    for bad in [(8, 3, 1, 1), (8, 2, 0, 1), (8, 2, 1, 0), (0, 1, 1, 1)]:
        with pytest.raises(nolo.NoloError) as e:
            nolo.nolo_sim_straggler(*bad, 1.0, 0.5, 1, 0)
        assert e.value.status == nolo.NOLO_EINVAL


def test_scratch_is_kept_and_bounded(nolo):
    """What is kept stays below 64 MB however large and small calls follow each other, and the largest of growing
    calls is kept (the driver hands memory out in pieces of 2 MB)."""
    import torch

    def call(mb):
        nolo.nolo_sim_tree_allreduce(2, 0.0, 0.5, (mb << 17) - 1000, 1)

    def give_back():
        nolo.nolo_destroy(nolo.nolo_create(2, 1, 8, 1, 0.5, 0.7, 0.5))
        torch.cuda.synchronize()

    call(1)
    give_back()
    free = torch.cuda.mem_get_info()[0]
    for small in (1, 2, 3):
        call(40)
        call(small)
        assert free - torch.cuda.mem_get_info()[0] <= (64 + 8) << 20
    give_back()
    for mb in (1, 2, 4, 8, 16, 32, 48):
        call(mb)
        assert free - torch.cuda.mem_get_info()[0] <= (64 + 8) << 20
    kept = torch.cuda.mem_get_info()[0]
    assert free - kept >= 48 << 20
    for mb in (48, 3, 48, 1, 2, 48):
        call(mb)
        assert torch.cuda.mem_get_info()[0] == kept
    give_back()
    assert free - torch.cuda.mem_get_info()[0] <= 4 << 20

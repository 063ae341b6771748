"""Kernels and rules for states with few columns and for small simulations, at the sizes where they change."""

import numpy as np
import pytest
import torch

from oracle import latency_oracle as L
from oracle import nolo_oracle as O
from paper_2506_10911_b200 import synth
from tests.helpers import to_np
from tests.test_gpu_magnitudes import step_and_compare

pytestmark = pytest.mark.gpu
HP = (0.5, 0.7, 0.5)


@pytest.fixture(scope="module")
def nolo():
    from paper_2506_10911_b200 import binding
    return binding


# All members at once up to 592 CTAs of 32 columns (n <= 128) or 296 of 16 columns (n <= 1024), else two passes: both
# sides of each line, for every shape whose order of the sums the former keeps.
LINES = [(12, 12, 592 * 32), (24, 12, 296 * 32), (24, 24, 592 * 32), (32, 32, 592 * 32), (64, 64, 592 * 32), (96, 96, 592 * 32),
         (128, 128, 592 * 32), (129, 129, 296 * 16), (224, 224, 296 * 16), (225, 225, 296 * 16), (641, 641, 296 * 16),
         (1024, 1024, 296 * 16)]


@pytest.mark.parametrize("W,n,P", LINES + [(W, n, P + 3) for W, n, P in LINES] + [
    (9, 9, 4), (32, 32, 1), (64, 64, 31), (40, 40, 130), (128, 128, 33), (130, 130, 5), (225, 225, 17), (1024, 1024, 1000), (2050, 1025, 150)])
@pytest.mark.parametrize("bf16", [False, True])
def test_outer_step_shapes(nolo, W, n, P, bf16):
    step_and_compare(nolo, W, n, P, torch.bfloat16 if bf16 else torch.float32, HP, seed=n + P)


@pytest.mark.parametrize("W,n,P", LINES)
@pytest.mark.parametrize("bf16", [False, True])
def test_bits_do_not_depend_on_the_number_of_columns(nolo, W, n, P, bf16):
    """The same columns in a state on either side of the line: the sums are added in the same order."""
    got = []
    state = synth.make_state(W, P + 64, n, torch.bfloat16 if bf16 else torch.float32)
    for cols in (P, P + 64):
        dev = [x.cuda() for x in state]
        h = nolo.nolo_create(W, n, cols, 1, *HP)
        nolo.nolo_bind_state(h, *dev)
        nolo.nolo_outer_step(h, 5, 6)
        torch.cuda.synchronize()
        nolo.nolo_destroy(h)
        got.append([x[:, :P] for x in dev])
    assert all(torch.equal(a, b) for a, b in zip(*got))


# A thread per quad or the members staged in pieces of 8 or 32 quads, in one to many stages of 64 or 16 rows.
@pytest.mark.parametrize("W,n,P", [(5, 5, 3), (7, 7, 1030), (15, 15, 2051), (16, 16, 4096), (63, 63, 517), (64, 64, 514), (65, 65, 4097),
                                   (130, 130, 6), (24, 12, 80_003), (64, 32, 40_001), (128, 128, 20_003),
                                   (17, 17, 4 * 4736 + 1), (34, 17, 4 * 2369), (1024, 1024, 9475), (2049, 2049, 260), (193, 193, 30_002), (569, 569, 2)])
def test_subgroup_means_of_few_columns(nolo, W, n, P):
    phi, theta, delta = synth.make_state(W, P, n, pad_value=float("nan"))
    dev = [x.cuda() for x in (phi, theta, delta)]
    mean = torch.full((W // n, synth.padded_stride(P, 8)), float("nan"), dtype=torch.float64, device="cuda")
    h = nolo.nolo_create(W, n, P, 1, *HP)
    nolo.nolo_bind_state(h, *dev)
    nolo.nolo_bind_prepared(h, mean)
    nolo.nolo_outer_prepare(h, 3, 3)
    got = mean.cpu().numpy()
    nolo.nolo_destroy(h)
    x = to_np(phi)[:, :P]
    # float32 pairs hold about 46 bits of a sum of n values
    np.testing.assert_allclose(got[:, :P], O.subgroup_mean_phi(x, O.draw_groups(3, 3, W, n), n), rtol=1e-12,
                               atol=1e-12 * float(np.abs(x).max()))
    assert np.isnan(got[:, P:]).all()


@pytest.mark.parametrize("W,n", [(5, 5), (16, 16), (17, 17), (34, 17), (32, 32), (64, 64), (96, 48), (255, 255), (256, 256), (1024, 1024), (2500, 1250)])
def test_subgroup_means_do_not_depend_on_the_number_of_columns(nolo, W, n):
    """A state cut by columns has the means of the whole, bit for bit: 8 quads, and both sides of each line."""
    groups = W // n
    few, narrow = 148 * (192 if n < 32 else 512) // groups, 148 * 32 // groups
    sizes = [32, 4 * narrow, 4 * narrow + 4, 4 * few, 4 * few + 4]
    cols = max(sizes)
    phi = 0.02 * torch.randn(W, synth.padded_stride(cols), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    z, d = torch.zeros_like(phi), torch.zeros_like(phi)
    got = []
    for P in sizes:
        mean = torch.full((groups, synth.padded_stride(P, 8)), float("nan"), dtype=torch.float64, device="cuda")
        h = nolo.nolo_create(W, n, P, 1, *HP)
        nolo.nolo_bind_state(h, phi, z, d)
        nolo.nolo_bind_prepared(h, mean)
        nolo.nolo_outer_prepare(h, 3, 3)
        torch.cuda.synchronize()
        nolo.nolo_destroy(h)
        got.append(mean)
    whole = got[sizes.index(cols)]
    for P, mean in zip(sizes, got):
        assert torch.equal(mean[:, :P], whole[:, :P])


@pytest.mark.parametrize("W,P", [(63, 1024 * 147), (64, 1024 * 147), (64, 1024 * 295 + 1), (16, 1024 * 148), (15, 1024 * 100 + 3)])
def test_divergence_in_parts(nolo, W, P):
    gen = torch.Generator().manual_seed(W)
    phi = 0.02 * torch.randn(1, synth.padded_stride(P), generator=gen) + 1e-3 * torch.randn(W, synth.padded_stride(P), generator=gen)
    dev = phi.cuda()
    h = nolo.nolo_create(W, 1, P, 1, *HP)
    nolo.nolo_bind_state(h, dev, torch.zeros_like(dev), torch.zeros_like(dev))
    got = nolo.nolo_divergence(h)
    nolo.nolo_destroy(h)
    std = phi[:, :P].double().std(0, correction=0)
    # a float32 variance per parameter: a few roundings of 2^-24 each
    assert got == pytest.approx((float(std.mean()), float(std.square().mean().sqrt())), rel=1e-6)


# 4, 16 and 32 parts, the last four workers of a part complete or not.
@pytest.mark.parametrize("W,P", [(16, 100_000), (24, 100_000), (32, 50_000), (64, 100_000), (63, 150_000), (64, 390_625), (300, 200_000),
                                 (1000, 100_000), (1024, 24_414)])
def test_divergence_in_parts_keeps_its_accuracy(nolo, W, P):
    """The deviations' roundings of each parameter, 2e-7 root mean square here, cancel in the mean over the parameters (below 1e-9
    left).  What does not cancel is a drift of sums of many terms of one sign: below a twelfth of a unit of 2^-24 as long as
    few terms follow each other (8e-9 with 16 workers one after the other)."""
    gen = torch.Generator().manual_seed(W)
    phi = 0.02 * torch.randn(1, synth.padded_stride(P), generator=gen) + 1e-3 * torch.randn(W, synth.padded_stride(P), generator=gen)
    dev = phi.cuda()
    h = nolo.nolo_create(W, 1, P, 1, *HP)
    nolo.nolo_bind_state(h, dev, torch.zeros_like(dev), torch.zeros_like(dev))
    got = nolo.nolo_divergence(h)
    nolo.nolo_destroy(h)
    std = torch.cat([x.double().std(0, correction=0) for x in dev[:, :P].split(50_000, 1)])
    assert got == pytest.approx((float(std.mean()), float(std.square().mean().sqrt())), rel=5e-9)


# Lanes per trial from 1 to 32 (many trials take few), subtrees of 0 to 32 leaf blocks per lane.
@pytest.mark.parametrize("W", [2, 4, 8, 32, 64, 128, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("many", [1, 70_000])
def test_tree_lanes(nolo, W, many):
    trials = max(1, many * 2 // W)
    *_, per = nolo.nolo_sim_tree_allreduce(W, 0.1, 0.9, trials, 17, return_trials=True)
    count = min(trials, max(1, 512 // W))
    assert per.shape == (trials,) and (per > 0).all()
    for first in {0, trials - count}:
        want = [_tree(W, s, 0.1, 0.9, 17) for s in range(first, first + count)]
        np.testing.assert_allclose(per[first:first + count], want, rtol=1e-11)


# 64 to 256 lanes, of several warps, in one round and several; the last trials of a CTA missing.
@pytest.mark.parametrize("W,trials", [(128, 148), (256, 300), (512, 1), (1024, 5), (1024, 601), (2048, 149), (2048, 1593), (4096, 3), (4096, 90),
                                      (4096, 1501)])
@pytest.mark.parametrize("sigma", [0.9, 90.0])
def test_tree_lanes_of_several_warps(nolo, W, trials, sigma):
    mean, _, per = nolo.nolo_sim_tree_allreduce(W, 0.1, sigma, trials, 17, return_trials=True)
    assert per.shape == (trials,) and (per > 0).all() and mean == pytest.approx(per.mean(), rel=1e-13)
    for first in {0, trials // 2, max(0, trials - 3)}:
        count = min(3, trials - first)
        want = [_tree(W, s, 0.1, sigma, 17) for s in range(first, first + count)]
        np.testing.assert_allclose(per[first:first + count], want, rtol=1e-11)


def _tree(W, trial, mu, sigma, seed):
    """Completion of one trial, level by level from the oracle's message times."""
    up, down = (L.message_times(W, trial, phase, mu, sigma, seed) for phase in (0, 1))
    ready = np.zeros(2 * W)
    for node in range(W - 1, 0, -1):
        ready[node] = max(ready[2 * node] + up[2 * node], ready[2 * node + 1] + up[2 * node + 1])
    at = np.zeros(2 * W)
    at[1] = ready[1]
    for node in range(2, 2 * W):
        at[node] = at[node // 2] + down[node]
    return at[W:].max()


# Results of up to 2^17 values are written to page-locked memory by the kernel, others copied.
@pytest.mark.parametrize("trials", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1])
def test_results_at_the_size_where_they_are_copied(nolo, trials):
    mean, _, per = nolo.nolo_sim_tree_allreduce(2, 0.1, 0.6, trials, 5, return_trials=True)
    *_, few = nolo.nolo_sim_tree_allreduce(2, 0.1, 0.6, 50, 5, return_trials=True)
    assert np.array_equal(per[:50], few) and (per > 0).all() and mean == pytest.approx(per.mean(), rel=1e-13)
    *_, per = nolo.nolo_sim_straggler(1, 1, 1, 1, 0.1, 0.6, trials // 2, 5, return_trials=True)
    *_, few = nolo.nolo_sim_straggler(1, 1, 1, 1, 0.1, 0.6, 50, 5, return_trials=True)
    assert np.array_equal(per[:50], few) and (per > 0).all()


# One subgroup of all workers; partitions of 4 to 32 lanes each; pairs and other subgroups; the last
# block of an item with one to four inner steps.
@pytest.mark.parametrize("W,n,H,T,trials", [
    (3, 3, 5, 40, 3), (64, 64, 6, 33, 2), (4096, 4096, 2, 3, 2), (4, 2, 7, 37, 9), (5, 1, 3, 4, 7), (8, 4, 4, 9, 3), (9, 3, 1, 5, 2),
    (16, 2, 2, 9, 5), (17, 17, 4, 3, 2), (15, 5, 3, 9, 3), (32, 8, 2, 5, 2), (256, 8, 2, 6, 2), (252, 7, 2, 6, 2), (258, 6, 2, 3, 1), (64, 2, 9, 8, 3), (66, 2, 10, 7, 2), (1024, 8, 3, 5, 1), (1026, 2, 3, 6, 1), (2048, 1, 2, 3, 1),
])
def test_straggler_rules(nolo, W, n, H, T, trials):
    *_, per = nolo.nolo_sim_straggler(W, n, H, T, 0.4, 0.8, trials, 21, return_trials=True)
    np.testing.assert_allclose(per, L.sim_straggler(W, n, H, T, 0.4, 0.8, trials, 21), rtol=1e-11)
    if n == W:
        assert np.array_equal(per[:, 0], per[:, 1])


# One slab (the first five) and several, of 2^21 - 2^12 work sums, from which pairs, the members of small subgroups, shared subgroups, more than
# 1024 workers and one subgroup of all go on.
@pytest.mark.parametrize("W,n,H,T,trials", [
    (4, 2, 30, 250, 300), (5, 5, 9, 250, 300), (16, 2, 130, 112, 160), (63, 3, 6, 61, 80), (3, 3, 13, 90, 1200),
    (64, 64, 40, 37, 900), (1024, 1024, 1, 5, 900), (512, 2, 2, 9, 700), (256, 8, 2, 40, 300), (252, 7, 2, 40, 300),
    (15, 3, 2, 100, 1500), (1024, 8, 2, 5, 900), (1024, 32, 2, 3, 2000), (288, 9, 1, 30, 300), (2048, 2, 2, 4, 600)])
def test_straggler_slabs_and_shared_rows(nolo, W, n, H, T, trials):
    *_, per = nolo.nolo_sim_straggler(W, n, H, T, 0.4, 0.8, trials, 21, return_trials=True)
    for first in (0, trials // 2, trials - 2):
        np.testing.assert_allclose(per[first:first + 2], L.sim_straggler(W, n, H, T, 0.4, 0.8, 2, 21, first), rtol=1e-11)
    assert (per[:, 1] <= per[:, 0] * (1 + 1e-15)).all() and (per > 0).all()


def test_the_largest_scratch_of_stragglers_is_kept(nolo):
    """One worker, two iterations and 1 046 528 trials need the most: 67.0e6 bytes, below the 2^26 that are kept (the driver hands memory
    out in pieces of 2 MB)."""
    def give_back():
        nolo.nolo_destroy(nolo.nolo_create(2, 1, 8, 1, *HP))
        torch.cuda.synchronize()

    nolo.nolo_sim_straggler(1, 1, 1, 1, 0.0, 0.5, 10, 1)
    give_back()
    free = torch.cuda.mem_get_info()[0]
    nolo.nolo_sim_straggler(1, 1, 1, 2, 0.0, 0.5, 1_046_528, 1)
    assert 64 << 20 >= free - torch.cuda.mem_get_info()[0] >= 62 << 20
    give_back()
    assert free - torch.cuda.mem_get_info()[0] <= 4 << 20


# Many trials leave a slab few iterations: units of 256 items lie across trials where one trial does not fill them.
@pytest.mark.parametrize("W,n,H,T,trials", [(64, 2, 6, 9, 4000), (100, 4, 5, 3, 9000), (257, 257, 3, 2, 7000), (65, 5, 9, 1, 3000),
                                            (64, 64, 130, 2, 17_000), (1000, 8, 2, 1, 300), (300, 10, 34, 2, 900), (128, 8, 3, 3, 31),
                                            (4, 2, 29, 1, 9000), (5, 1, 2, 20, 70_000), (63, 9, 30, 2, 40_000)])
@pytest.mark.parametrize("sigma", [0.8, 90.0])
def test_straggler_units_across_trials(nolo, W, n, H, T, trials, sigma):
    *_, per = nolo.nolo_sim_straggler(W, n, H, T, 0.4, sigma, trials, 21, return_trials=True)
    for first in (0, trials // 2, trials - 2):
        want = L.sim_straggler(W, n, H, T, 0.4, sigma, 2, 21, first)
        # (an exponent of 8.7 sigma has units of 2^-53 times that)
        np.testing.assert_allclose(per[first:first + 2], want, rtol=1e-11)


def test_calls_of_different_sizes_from_several_threads(nolo):
    """The kernels' shared memory depends on the sizes; what one call sets up must do for the others.  Every call gives what
    it gives when nothing else runs."""
    import threading
    trees, stragglers, states = [(1024, 300), (64, 300), (4096, 20), (2048, 20)], [(1024, 512), (100, 10), (64, 2), (1024, 2)], [130, 1024, 256, 700]

    def calls(k):
        """The simulations of every turn and, at the end, the state."""
        stream = torch.cuda.Stream()
        dev = [x.cuda() for x in synth.make_state(states[k], 900, k)]
        h = nolo.nolo_create(states[k], states[k], 900, 1, *HP)
        torch.cuda.synchronize()
        nolo.nolo_bind_state(h, *dev, stream=stream)
        sims = []
        for turn in range(30):
            sims += [nolo.nolo_sim_tree_allreduce(trees[k][0], 0.0, 1.0, trees[k][1], 3, stream, return_trials=True)[2],
                     nolo.nolo_sim_straggler(*stragglers[k], 3, 4, 0.0, 0.5, 5, 3, stream, return_trials=True)[4]]
            nolo.nolo_outer_step(h, 1, turn)
        stream.synchronize()
        nolo.nolo_destroy(h)
        return sims, [x.cpu() for x in dev]

    want = [calls(k) for k in range(4)]
    bad = []

    def work(k):
        try:
            sims, state = calls(k)
            if not all(np.array_equal(a, b) for a, b in zip(sims, want[k][0])):
                bad.append(f"simulations {k}")
            if not all(torch.equal(a, b) for a, b in zip(state, want[k][1])):
                bad.append(f"state {k}")
        except Exception as e:
            bad.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


# Copies draw for themselves up to 1 GB, of blocks that are no multiple of 32 bytes 100 MB, for up to 8 replicas and tiles of 16 KB that
# are filled to four fifths (128 and 64 MB otherwise): both sides of each line, E float32 elements in each of 2 boundaries x K x W.
@pytest.mark.parametrize("W,K,E,draws", [
    (8, 1, 1 << 24, True), (8, 1, (1 << 24) + 8, False), (8, 1, 50 * 32768 - 1, True), (8, 1, 50 * 32768 + 1, False),
    (9, 1, 932_067, True), (9, 1, 932_069, False), (9, 1, 1_864_128, True), (9, 1, 1_864_136, False), (7, 1, 3_000_000, True), (3, 1, 4_000_001, True),
    (8, 3000, 1000, False), (4, 8000, 512, True), (4, 8200, 512, False), (8, 700, 3280, True), (8, 700, 3272, False), (2, 1000, 4104, True),
    (6, 700, 4104, False), (8, 300, 3277, True), (8, 400, 3277, True), (8, 400, 3275, False), (3, 900, 4099, False), (5, 2, 1_200_001, True)])
def test_routing_at_the_sizes_where_copies_stop_drawing(nolo, W, K, E, draws):
    stages = 3
    acts = torch.randint(-2**31, 2**31 - 1, (stages - 1, W, K, E), dtype=torch.int32, device="cuda")
    out, back = torch.zeros_like(acts), torch.zeros_like(acts)
    h = nolo.nolo_create(W, 1, 8, stages, *HP)
    nolo.nolo_bind_route(h, W * K, E, out.view(torch.float32), True)
    before = nolo.nolo_launch_count(h)
    nolo.nolo_route(h, 11, 3, acts.view(torch.float32))
    assert nolo.nolo_launch_count(h) - before == (1 if draws else 2)
    table = torch.from_numpy(O.draw_route(11, 3, stages, W, K, per_microbatch=True)).long()
    assert np.array_equal(nolo.nolo_get_route(h), table.numpy())
    k = torch.arange(K)[:, None].cuda()
    for b in range(stages - 1):
        from_replica = table[b].cuda()                          # [K][W]
        for r in range(W):
            assert torch.equal(out[b, r], acts[b][from_replica[:, r], k[:, 0]])
    nolo.nolo_route_backward(h, 11, 3, out.view(torch.float32), back.view(torch.float32))
    torch.cuda.synchronize()
    assert torch.equal(back, acts)
    nolo.nolo_destroy(h)

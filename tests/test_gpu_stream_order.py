"""Calls that follow each other in a stream without any wait between them."""

import numpy as np
import pytest
import torch

from oracle import nolo_oracle as O
from paper_2506_10911_b200 import synth
from tests.helpers import to_np

pytestmark = pytest.mark.gpu

F = tuple(float(np.float32(x)) for x in (0.5, 0.7, 0.5))


@pytest.fixture(scope="module")
def nolo():
    from paper_2506_10911_b200 import binding
    return binding


def both(nolo, W, n, P, act):
    """The state after act(handle, step) for a train of steps, and after the same steps waited for one by one."""
    states = []
    for wait in (False, True):
        state = [x.cuda() for x in synth.make_state(W, P, 4)]
        h = nolo.nolo_create(W, n, P, 1, *F)
        nolo.nolo_bind_state(h, *state)
        mean = torch.zeros((W // n, state[0].shape[1]), dtype=torch.float64, device="cuda")
        nolo.nolo_bind_prepared(h, mean)
        for step in range(12):
            act(h, step)
            if wait:
                torch.cuda.synchronize()
                assert np.array_equal(nolo.nolo_get_groups(h), O.draw_groups(8, step, W, n))
        assert np.array_equal(nolo.nolo_get_groups(h), O.draw_groups(8, 11, W, n))
        nolo.nolo_destroy(h)
        states.append((*state, mean))
    return states


# More than 32 workers: the table is drawn by a kernel ahead of each step.  Grids of several times what the chip
# holds, so that CTAs of consecutive kernels share SMs.
@pytest.mark.parametrize("W,n,P", [(64, 2, 60_000), (40, 8, 90_003), (60, 20, 50_000), (128, 128, 40_000)])
def test_tables_drawn_ahead_are_those_of_their_step(nolo, W, n, P):
    a, b = both(nolo, W, n, P, lambda h, step: nolo.nolo_outer_step(h, 8, step))
    for x, y in zip(a, b):
        assert torch.equal(x, y)


@pytest.mark.parametrize("W,n,P", [(64, 2, 60_000), (40, 8, 90_003), (60, 20, 50_000), (8, 2, 300_000)])
def test_prepared_means_are_those_of_their_step(nolo, W, n, P):
    def act(h, step):
        nolo.nolo_outer_prepare(h, 8, step)
        nolo.nolo_outer_step_prepared(h, 8, step)
    a, b = both(nolo, W, n, P, act)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


@pytest.mark.parametrize("E", [20_480, 20_483])
@pytest.mark.parametrize("pm", [False, True])
def test_routes_are_those_of_their_step(nolo, E, pm):
    """There and back again: what one call writes the next reads, with a table that changes every step."""
    S, R, K = 3, 40, 4
    acts = synth.make_acts(S - 1, R, K, E, 2, torch.bfloat16).cuda()
    a, b = acts.clone(), torch.zeros_like(acts)
    h = nolo.nolo_create(R, 1, 8, S, *F)
    nolo.nolo_bind_route(h, R * K, E, b, per_microbatch=pm)
    want = to_np(acts)
    for step in range(8):
        nolo.nolo_route(h, 9, step, a)                              # a -> b
        nolo.nolo_route_backward(h, 9, 100 + step, b, a)            # b -> a, by another table
        want = O.route_backward(O.route_forward(want, O.draw_route(9, step, S, R, K, pm)),
                                O.draw_route(9, 100 + step, S, R, K, pm))
    assert np.array_equal(to_np(a), want)
    nolo.nolo_destroy(h)

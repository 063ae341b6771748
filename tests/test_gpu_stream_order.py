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


FOREIGN = r"""
#include <cuda_runtime.h>
// Reads samples of x ahead of its wait, as kernels do with weights.
__global__ void early_reader(const volatile float* x, long long stride, float* seen) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    seen[i] = x[i * stride];
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
extern "C" int launch_early_reader(const float* x, long long stride, float* seen, int blocks, void* stream) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(32);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, early_reader, (const volatile float*)x, stride, seen);
}
"""


@pytest.fixture(scope="module")
def early_reader(tmp_path_factory):
    import ctypes
    import subprocess
    from paper_2506_10911_b200 import build
    d = tmp_path_factory.mktemp("foreign")
    (d / "foreign.cu").write_text(FOREIGN)
    subprocess.run([build.find_nvcc(), *build.NVCC_FLAGS, "-o", str(d / "foreign.so"), str(d / "foreign.cu")], check=True)
    fn = ctypes.CDLL(str(d / "foreign.so")).launch_early_reader
    fn.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    return fn


@pytest.mark.parametrize("W,n", [(8, 2), (64, 8), (20, 20), (128, 128)])
@pytest.mark.parametrize("routed", [False, True])
def test_a_callers_kernel_sees_the_new_weights_ahead_of_its_wait(nolo, early_reader, W, n, routed):
    """Also with a routing call between the step and the caller's kernel."""
    P, blocks = (1 << 25) // W // 8 * 8, 64
    phi = torch.empty((W, P), device="cuda").uniform_(-0.05, 0.05)
    theta = torch.full_like(phi, 7.0)                       # fast weights far from anything a step leaves
    h = nolo.nolo_create(W, n, P, 2, *F)
    nolo.nolo_bind_state(h, phi, theta, torch.zeros_like(phi))
    acts = torch.zeros((1, W, 1, 1 << 12), device="cuda")
    out = torch.zeros_like(acts)
    nolo.nolo_bind_route(h, W, 1 << 12, out)
    stride = W * P // (blocks * 32)
    stream = torch.cuda.current_stream().cuda_stream
    for step in range(4):
        theta.fill_(7.0)
        seen = torch.empty(blocks * 32, device="cuda")
        nolo.nolo_outer_step(h, 1, step)
        if routed:
            nolo.nolo_route(h, 1, step, acts)
        assert early_reader(theta.data_ptr(), stride, seen.data_ptr(), blocks, stream) == 0
        assert torch.equal(seen, theta.view(-1)[::stride][:blocks * 32])
        assert not bool((seen == 7.0).any())
    nolo.nolo_destroy(h)


@pytest.mark.parametrize("W,P", [(8, 5000), (40, 70_003)])
def test_captured_calls_replay_as_they_run(nolo, W, P):
    """Both ways round, the step, the prepared step and the same from a second stream that joins in, captured into
    a graph: tables drawn inside the kernels (8 workers) and ahead of them (40)."""
    K, E, n = 2, 3001, 2
    state = [x.cuda() for x in synth.make_state(W, P, 4)]
    acts = synth.make_acts(1, W, K, E, 2, torch.bfloat16).cuda()
    results = []
    for captured in (False, True):
        mine = [x.clone() for x in state]
        out, back = torch.zeros_like(acts), torch.zeros_like(acts)
        mean = torch.zeros((W // n, mine[0].shape[1]), dtype=torch.float64, device="cuda")
        side, other = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()

        def calls():
            for step in range(3):
                nolo.nolo_route(h, 3, step, acts)
                nolo.nolo_route_backward(h, 3, step, out, back)
                nolo.nolo_outer_step(h, 3, step)
                other.wait_stream(side)
                with torch.cuda.stream(other):
                    mine[2].mul_(0.5)
                side.wait_stream(other)
                nolo.nolo_outer_prepare(h, 3, step + 100)
                nolo.nolo_outer_step_prepared(h, 3, step + 100)

        h = nolo.nolo_create(W, n, P, 2, *F)
        nolo.nolo_bind_state(h, *mine, stream=side)
        nolo.nolo_bind_prepared(h, mean)
        nolo.nolo_bind_route(h, W * K, E, out)
        with torch.cuda.stream(side):
            if captured:
                graph = torch.cuda.CUDAGraph()
                graph.capture_begin()
                calls()
                graph.capture_end()
                graph.replay()
            else:
                calls()
        torch.cuda.synchronize()
        assert torch.equal(back, acts)
        results.append((*mine, out, mean))
        nolo.nolo_destroy(h)
    for x, y in zip(*results):
        assert torch.equal(x, y)

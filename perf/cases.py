"""The work that users of this library have it do, as cases that can be timed and compared.

A case names a kind of call and its sizes.  ``listed()`` holds twelve that stand for the whole
range, ``draw()`` gives further ones of the same ranges, ``prepare()`` builds what a program has in
hand before the call (state or activations on the device, the bound handle), ``run()`` makes one
pass through the public entry points and ``work()`` states the bytes or operations that a pass
cannot do without.

Kinds:
  outer       one outer step (Eq. 1-3), through the handle or the allocation-free entry point
  step        the data-parallel part of one training step with pipeline stages: outer step, forward
              routing, backward routing
  split       the outer step in two phases: subgroup means of the slow weights, then the step
  route       routing of all stage boundaries, forward and backward
  boundary    routing of one stage boundary (what one pipeline stage does)
  divergence  the replica-divergence metric (Fig. 3b)
  host        outer step and forward routing of state that lives in page-locked host memory
  straggler   Monte-Carlo cost of the global barrier (Fig. 5b)
  tree        Monte-Carlo tree all-reduce (Fig. 5a)
"""

from __future__ import annotations

import math

import torch

from paper_2506_10911_b200 import binding as nolo
from paper_2506_10911_b200 import synth

ALPHA, BETA, GAMMA = 0.5, 0.7, 0.5
THETA = {"f32": torch.float32, "bf16": torch.bfloat16}


# ---- the cases ----------------------------------------------------------------------------------

def _outer(W, n, P, theta, drift="normal", static=False):
    return {"kind": "outer", "W": W, "n": n, "P": P, "theta": theta, "drift": drift, "static": static}


def _step(W, n, P, theta, stages, K, E, act):
    return {"kind": "step", "W": W, "n": n, "P": P, "theta": theta, "stages": stages, "K": K, "E": E, "act": act,
            "per_microbatch": False}


def _split(W, n, P, theta, drift="normal"):
    return {"kind": "split", "W": W, "n": n, "P": P, "theta": theta, "drift": drift}


def _route(kind, W, stages, K, E, act, per_microbatch):
    return {"kind": kind, "W": W, "stages": stages, "K": K, "E": E, "act": act, "per_microbatch": per_microbatch}


def _divergence(W, P):
    return {"kind": "divergence", "W": W, "P": P}


def _host(W, n, P, theta, stages, K, E, act):
    return {"kind": "host", "W": W, "n": n, "P": P, "theta": theta, "stages": stages, "K": K, "E": E, "act": act,
            "per_microbatch": False}


def _straggler(W, n, H, T, trials):
    return {"kind": "straggler", "W": W, "n": n, "H": H, "T": T, "mu": 1.0, "sigma": math.sqrt(0.5), "trials": trials}


def _tree(W, sigma, trials):
    return {"kind": "tree", "W": W, "mu": 0.0, "sigma": sigma, "trials": trials}


def listed():
    return [
        # A toy model or one small parameter group: the call's latency is everything.
        dict(_outer(4, 2, 1 << 16, "f32"), name="outer_small"),
        # The first benchmark configuration: four replicas of a million parameters in pairs, eight
        # micro-batches of 2 x 128 x 256 float32 activations over two stages.
        dict(_step(4, 2, 1 << 20, "f32", 2, 2, 2 * 128 * 256, "f32"), name="step_4x1M"),
        # The 125M decoder, sixteen replicas in pairs, bfloat16 fast weights: the ordinary outer step.
        dict(_outer(16, 2, synth.model_params("125M"), "bf16"), name="outer_125M_pairs"),
        # Middle-sized subgroups of a shard whose parameter count is not a multiple of anything.
        dict(_outer(60, 20, 1_000_003, "f32"), name="outer_ragged_n20"),
        # DiLoCo mode: one subgroup of all workers, at the widest size of the benchmark.
        dict(_outer(1024, 1024, 786_432, "bf16"), name="outer_diloco_1024"),
        # The step in two phases for subgroups of eight, heavy-tailed drift (the worker sweep's
        # largest subgroup at a quarter of its parameters).
        dict(_split(32, 8, 1 << 24, "f32", "student_t3"), name="split_32x16M_n8"),
        # Routing of 32 micro-batches of 4 x 2048 x 4096 bfloat16 activations over four stages.
        dict(_route("route", 8, 4, 4, 4 * 2048 * 4096, "bf16", False), name="route_32x4x2048x4096"),
        # Routing of odd-sized activations, every micro-batch with a permutation of its own.
        dict(_route("route", 8, 3, 4, 3 * 257 * 769, "bf16", True), name="route_ragged"),
        # The divergence metric as a training loop logs it: a layer's worth of parameters of sixteen replicas.
        dict(_divergence(16, synth.layer_params(768, 3072)), name="divergence_layer"),
        # State and activations in page-locked host memory, one decoder layer and a quarter million more.
        dict(_host(8, 2, synth.layer_params(768, 3072) + 250_000, "bf16", 2, 2, 2 * 512 * 768, "bf16"), name="host_8x7M"),
        # Fig. 5b at its largest size with the trials of the command-line default.
        dict(_straggler(1024, 2, 100, 250, 148), name="straggler_1024"),
        # Fig. 5a at its largest size with 20 000 trials.
        dict(_tree(1024, 1.0, 20_000), name="tree_1024"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _params(rng, lo, hi):
    """A parameter count: half of them odd, some a multiple of a tile, the rest as they come."""
    P = _log(rng, lo, hi)
    how = rng.random()
    return max(1, P | 1 if how < 0.5 else P & ~1023 if how < 0.75 else P)


def _subgroup(rng, W):
    """Pairs are what the method is for; DiLoCo mode (all workers) and every divisor also occur."""
    divisors = [d for d in range(2, W + 1) if W % d == 0] or [1]
    how = rng.random()
    return divisors[0] if how < 0.35 else W if how > 0.85 else rng.choice(divisors)


def draw(rng):
    kind = rng.choices(["outer", "step", "split", "route", "boundary", "divergence", "host", "straggler", "tree"],
                       [36, 10, 8, 9, 4, 8, 9, 8, 8])[0]
    if kind in ("outer", "split", "step"):
        W = rng.choice([2, 4, 6, 8, 8, 12, 16, 16, 24, 32, 32, 48, 60, 64, 96, 128, 128, 256, 512, 1024])
        most = {"outer": 1.6e9, "split": 6e8, "step": 3e8}[kind]          # worker-parameters
        P = _params(rng, max(1000, 1e5 / W), most / W)
        n, theta = _subgroup(rng, W), rng.choice(["f32", "bf16"])
        if kind == "outer":
            return _outer(W, n, P, theta, rng.choice(["normal", "student_t3"]), rng.random() < 0.2)
        if kind == "split":
            return _split(W, n, P, theta)
        W = min(W, 32)
        n = min(n, W) if W % min(n, W) == 0 else W
        return _step(W, n, P, theta, rng.choice([2, 3, 4]), rng.choice([1, 2, 4]), _log(rng, 4096, 1 << 21),
                     rng.choice(["f32", "bf16"]))
    if kind in ("route", "boundary"):
        W, stages, K = rng.choice([4, 6, 8, 16, 32]), rng.choice([2, 3, 4, 8]), rng.choice([1, 2, 4, 8])
        blocks = W * K * (stages - 1)
        E = _params(rng, 1000, min(1 << 25, 1.5e9 / blocks))
        return _route(kind, W, stages, K, E, rng.choice(["f32", "bf16"]), rng.random() < 0.4)
    if kind == "divergence":
        W = rng.choice([2, 4, 8, 16, 32, 64, 128, 1024])
        return _divergence(W, _params(rng, max(1000, 1e5 / W), 1.8e9 / W))
    if kind == "host":
        W = rng.choice([2, 4, 8, 16, 32])
        n = _subgroup(rng, W)
        K, E = rng.choice([1, 2, 4]), _log(rng, 4096, 1 << 20)
        return _host(W, n, _params(rng, 2e5 / W, 1e8 / W), rng.choice(["f32", "bf16"]), rng.choice([2, 3, 4]), K, E,
                     rng.choice(["f32", "bf16"]))
    if kind == "straggler":
        W = rng.choice([4, 16, 64, 100, 256, 512, 1024])
        H, T = rng.choice([10, 25, 50, 100]), rng.choice([50, 100, 250, 500])
        return _straggler(W, _subgroup(rng, W), H, T, _log(rng, 8, min(592, 3e9 / (W * H * T))))
    W = rng.choice([2, 4, 16, 64, 256, 1024])
    return _tree(W, rng.choice([0.1, 0.5, 1.0]), _log(rng, 1000, min(400_000, 4e7 / W)))


# ---- what a program has in hand ---------------------------------------------------------------------

def _state(c, seed):
    stride = synth.padded_stride(c["P"])
    phi = torch.zeros((c["W"], stride), dtype=torch.float32, device="cuda")
    theta = torch.zeros((c["W"], stride), dtype=THETA[c.get("theta", "f32")], device="cuda")
    delta = torch.zeros((c["W"], stride), dtype=torch.float32, device="cuda")
    synth.fill_state_(phi, theta, delta, c["P"], seed, c.get("drift", "normal"))
    return phi, theta, delta


def _handle(c):
    return nolo.nolo_create(c["W"], c.get("n", 1), c.get("P", 8), c.get("stages", 1), ALPHA, BETA, GAMMA)


def _acts(c, seed):
    return synth.make_acts(c["stages"] - 1, c["W"], c["K"], c["E"], seed, THETA[c["act"]], "cuda")


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def prepare(case, seed):
    c = case
    kind = c["kind"]
    s = {"case": c, "seed": seed, "step": 0}
    if kind in ("straggler", "tree"):
        torch.zeros(1, device="cuda")
        return s
    if kind == "divergence":
        # replicas that have stayed close to a common point
        stride = synth.padded_stride(c["P"])
        gen = torch.Generator(device="cuda").manual_seed(seed)
        base = torch.zeros(stride, device="cuda").normal_(0.0, synth.PHI_STD, generator=gen)
        phi = torch.empty((c["W"], stride), device="cuda").normal_(0.0, synth.DRIFT_STD, generator=gen).add_(base)
        h = _handle(c)
        # the metric reads the slow weights only; the other two buffers are what the handle is bound to
        theta = torch.empty((c["W"], stride), dtype=torch.bfloat16, device="cuda")
        delta = torch.empty((c["W"], stride), device="cuda")
        nolo.nolo_bind_state(h, phi, theta, delta)
        s.update(h=h)
        return s
    h = _handle(c) if not c.get("static") else None
    if "P" in c:
        state = _state(c, seed)
        s["state"] = state
        if h is not None:
            nolo.nolo_bind_state(h, *state)
    if kind == "split":
        s["mean"] = torch.zeros((c["W"] // c["n"], state[0].shape[1]), dtype=torch.float64, device="cuda")
        nolo.nolo_bind_prepared(h, s["mean"])
    if "stages" in c:
        acts = _acts(c, seed + 1)
        out = torch.zeros_like(acts)
        nolo.nolo_bind_route(h, c["W"] * c["K"], c["E"], out, c["per_microbatch"])
        s.update(acts=acts, out=out)
        if kind in ("step", "route"):
            s.update(grads=_acts(c, seed + 2), grads_out=torch.zeros_like(acts))
        if kind == "boundary":
            s["out_b"] = torch.zeros_like(acts[0])
        if kind == "host":
            s.update(h_state=[_pinned(x) for x in state], h_acts=_pinned(acts), h_out=_pinned(out))
    s["h"] = h
    return s


# ---- one pass -------------------------------------------------------------------------------------------

def run(state):
    s, c = state, state["case"]
    kind, seed = c["kind"], s["seed"]
    step = s["step"]
    s["step"] += 1
    if kind == "straggler":
        return nolo.nolo_sim_straggler(c["W"], c["n"], c["H"], c["T"], c["mu"], c["sigma"], c["trials"], seed + step,
                                       return_trials=True)
    if kind == "tree":
        return nolo.nolo_sim_tree_allreduce(c["W"], c["mu"], c["sigma"], c["trials"], seed + step, return_trials=True)
    h = s["h"]
    if kind == "outer":
        if c["static"]:
            nolo.nolo_outer_step_static(c["W"], c["n"], c["P"], ALPHA, BETA, GAMMA, *s["state"], seed, step)
        else:
            nolo.nolo_outer_step(h, seed, step)
        return s["state"]
    if kind == "step":
        nolo.nolo_route(h, seed, step, s["acts"])
        nolo.nolo_route_backward(h, seed, step, s["grads"], s["grads_out"])
        nolo.nolo_outer_step(h, seed, step)
        return (*s["state"], s["out"], s["grads_out"])
    if kind == "split":
        nolo.nolo_outer_prepare(h, seed, step)
        nolo.nolo_outer_step_prepared(h, seed, step)
        return (*s["state"], s["mean"])
    if kind == "route":
        nolo.nolo_route(h, seed, step, s["acts"])
        nolo.nolo_route_backward(h, seed, step, s["grads"], s["grads_out"])
        return s["out"], s["grads_out"]
    if kind == "boundary":
        b = c["stages"] - 2
        nolo.nolo_route_boundary(h, seed, step, b, s["acts"][b], s["out_b"])
        return s["out_b"]
    if kind == "divergence":
        return nolo.nolo_divergence(h)
    nolo.nolo_outer_step_host(h, seed, step, *s["h_state"])
    nolo.nolo_route_host(h, seed, step, s["h_acts"], s["h_out"], s["acts"])
    return (*s["h_state"], s["h_out"])


# ---- what a pass cannot do without ------------------------------------------------------------------------

# Operations of one log-normal time: a quarter of a Philox block (ten rounds of two 64 x 64 -> 128-bit
# products, four exclusive-ors and two additions, a wide product counted as four), half a logarithm,
# square root and sine-cosine pair, and one exponential (a polynomial of about ten terms each).
SIM_FLOPS_PER_SAMPLE = 75


def work(case):
    c = case
    kind = c["kind"]
    if kind == "straggler":
        return {"bytes": 16.0 * c["trials"], "flops": float(SIM_FLOPS_PER_SAMPLE) * c["W"] * c["H"] * c["T"] * c["trials"]}
    if kind == "tree":
        return {"bytes": 8.0 * c["trials"], "flops": float(SIM_FLOPS_PER_SAMPLE) * (4 * c["W"] - 4) * c["trials"]}
    moved, flops = 0.0, 0.0
    if kind == "divergence":
        return {"bytes": 4.0 * c["W"] * c["P"], "flops": 6.0 * c["W"] * c["P"]}
    if "P" in c:
        wp = float(c["W"]) * c["P"]
        moved += wp * (20 if c["theta"] == "bf16" else 24)
        flops += 10.0 * wp
        if kind == "split":
            moved += wp * 4 + 16.0 * wp / c["n"]       # slow weights read early, means written and read
    if "stages" in c:
        size = 2 if c["act"] == "bf16" else 4
        boundaries = 1 if kind == "boundary" else c["stages"] - 1
        directions = 2 if kind in ("step", "route") else 1
        moved += 2.0 * size * boundaries * c["W"] * c["K"] * c["E"] * directions
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("route", "boundary"):
        return "exact"
    if kind in ("straggler", "tree"):
        # float64 sums of up to 1e5 terms of functions that are good to one or two units in the last place:
        # times within 5e-16 of the float64 definition, standard errors of few trials within 2e-14
        return {"rel": 1e-13, "max": 1e-12}
    if kind == "divergence":
        # float32 variance per parameter, float64 sums: within 1.3e-8 of float64 in one order of the sums
        return {"rel": 2e-7}
    if case["theta"] == "bf16":
        # as below, and where float32 results straddle a bfloat16 rounding boundary theta moves by one unit
        # (2^-7 of the value at most): within 3.8e-5 and 7.8e-3 of float64
        return {"rel": 1.5e-4, "max": 1e-2}
    # float32 momentum and weights: within 4e-8 of float64, and within 5.4e-7 and 4.6e-6 where a step
    # nearly cancels the weights (the second step of a subgroup of all workers)
    return {"rel": 2e-6, "max": 2e-5}

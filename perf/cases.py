"""Workloads of the CORE library: what its users have it do, through its public entry points.

A case is one call (or the calls of one machine in one round) with everything a user's program already
holds - gradients or data matrices, the context, the least-squares handle, output buffers - made
beforehand by ``prepare``.  Kinds:

  round          ``core_round``: n simulated machines, G[n, d] on the device -> p̄[m], g̃[d]
  machine        one machine per GPU: ``core_project`` of its own gradient, ``core_aggregate`` of the
                 gathered messages, ``core_reconstruct``
  host           ``core_round_host``: the round with gradients and estimate in pinned host memory
  gd, agd        one iteration of CORE-GD / CORE-AGD on a distributed least-squares problem
  guarded        one iteration with the comparison step (a second evaluation of f, decided on the device)
  decentralized  one iteration in which gossip with the neighbours replaces the central machine

``listed`` holds the named cases, ``draw`` gives more of the same ranges, ``run`` is one pass, ``work``
the bytes and multiply-adds a pass cannot do without, ``tolerance`` what another correct implementation
of the same precision may differ by.
"""
from __future__ import annotations

import math

import torch

import core_inputs
from paper_2309_13307_b200 import binding

GENERATOR_SEED = 1
ROUND_KINDS = ("round", "machine", "host")
LS_KINDS = ("gd", "agd", "guarded", "decentralized")


def listed():
    return [
        # the smallest evaluation workload: a handful of kernels on 4096 coordinates, all latency
        {"name": "round tiny", "kind": "round", "n": 4, "d": 4096, "m": 16, "dtype": "f32", "dist": "normal", "pad": False},
        # an odd number of machines on a vector whose length is a multiple of nothing: rows packed back to
        # back, so that only the first is aligned; a number of vectors that is no power of two
        {"name": "round ragged", "kind": "round", "n": 5, "d": 1_000_003, "m": 100, "dtype": "f32", "dist": "normal", "pad": False},
        # the resnet50 workload: 8 machines, fp32 gradients of different scale
        {"name": "round resnet50", "kind": "round", "n": 8, "d": 25_557_032, "m": 256, "dtype": "f32", "dist": "scaled_normal", "pad": False},
        # 32 simulated machines at fp32, the largest count the paper trains a network with
        {"name": "round 32 machines", "kind": "round", "n": 32, "d": 10_000_000, "m": 1000, "dtype": "f32", "dist": "normal", "pad": False},
        # the gpt2small workload: 16 machines, heavy-tailed bf16 gradients, a long message
        {"name": "round gpt2small", "kind": "round", "n": 16, "d": 124_439_808, "m": 1024, "dtype": "bf16", "dist": "student_t3", "pad": False},
        # the longest vectors (the projection-dimension sweep of the benchmark at one of its m)
        {"name": "round sweep", "kind": "round", "n": 2, "d": 1_000_000_000, "m": 64, "dtype": "f32", "dist": "normal", "pad": False},
        # one rank of a machine-per-GPU deployment: its own bf16 gradient out, the common estimate back
        {"name": "machine", "kind": "machine", "n": 8, "d": 25_557_032, "m": 256, "dtype": "bf16", "dist": "normal", "pad": False},
        # gradients that live on the host (an offloaded optimiser): bound by the copies unless m is large
        {"name": "host", "kind": "host", "n": 8, "d": 4_000_000, "m": 64, "dtype": "f32", "dist": "normal", "pad": False},
        # the leastsq workload: the CORE-GD iteration whose trajectory the tests follow
        {"name": "gd leastsq", "kind": "gd", "n": 8, "rows": 2048, "d": 8192, "m": 64},
        # linear models on image-sized features over the paper's 50 machines, accelerated
        {"name": "agd 50 machines", "kind": "agd", "n": 50, "rows": 1200, "d": 784, "m": 64},
        # tall tabular data with few, oddly many features over 50 machines, with the comparison step
        {"name": "guarded tall", "kind": "guarded", "n": 50, "rows": 11620, "d": 54, "m": 16},
        # wide features, a ring of machines, twenty gossip rounds per iteration
        {"name": "decentralized wide", "kind": "decentralized", "n": 16, "rows": 256, "d": 20_000, "m": 64, "rounds": 20},
    ]


def _log_int(rng, low, high):
    return max(low, min(high, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    kind = rng.choice(ROUND_KINDS + LS_KINDS + ("round", "round"))
    if kind in ROUND_KINDS:
        case = {"kind": kind, "n": _log_int(rng, 1, 64), "m": _log_int(rng, 8, 4096),
                "dtype": rng.choice(("f32", "bf16")), "dist": rng.choice(("normal", "scaled_normal")),
                "pad": rng.random() < 0.25}
        size = 2 if case["dtype"] == "bf16" else 4
        rows = 1 if kind == "machine" else case["n"]
        # host buffers stay within 128 MB and device gradients within 8 GB; the Gaussians of a pass within
        # 3e10, a quarter of the largest listed case
        most = (128e6 if kind == "host" else 8e9) / (size * rows)
        high = int(min(most, 1e9, 3e10 / case["m"]))
        case["d"] = _log_int(rng, min(1000, high), high)
        return case
    case = {"kind": kind, "n": _log_int(rng, 2, 64), "m": _log_int(rng, 8, 256), "d": _log_int(rng, 32, 32768)}
    # data matrices of up to 512 MiB over all machines
    most = int((1 << 27) / (case["n"] * case["d"]))
    case["rows"] = _log_int(rng, 16, max(17, min(16384, most)))
    if kind == "decentralized":
        case["rounds"] = _log_int(rng, 4, 64)
    return case


def _prepare_round(case, seed):
    kind, n, d, m = case["kind"], case["n"], case["d"], case["m"]
    rows = 1 if kind == "machine" else n
    ld = (d + 7) // 8 * 8 if case["pad"] else d         # a padded leading dimension keeps every row aligned
    G = core_inputs.gradients(rows, d, seed=seed, dist=case["dist"], dtype=case["dtype"], device="cuda", ld=ld)
    core = binding.Core(GENERATOR_SEED, d, m)
    state = {"kind": kind, "core": core, "G": G}
    if kind == "host":
        store = torch.empty((n, ld), dtype=G.dtype, pin_memory=True)
        state["G"] = store[:, :d]
        state["G"].copy_(G)
        state["pbar"] = torch.empty(m, dtype=torch.float32, pin_memory=True)
        state["gtilde"] = torch.empty(d, dtype=torch.float32, pin_memory=True)
        return state
    core.core_reserve_workspace(rows, binding.CORE_BF16 if case["dtype"] == "bf16" else binding.CORE_F32)
    state["pbar"] = torch.empty(m, dtype=torch.float32, device="cuda")
    state["gtilde"] = torch.empty(d, dtype=torch.float32, device="cuda")
    if kind == "machine":
        # the other machines' messages, as the exchange left them; row 0 is this machine's
        state["P"] = torch.empty((1, m), dtype=torch.float32, device="cuda")
        state["P_all"] = core_inputs.gradients(n, m, seed=seed + 1_000_003, device="cuda") * math.sqrt(d)
    return state


def _prepare_ls(case, seed):
    n, d, m = case["n"], case["d"], case["m"]
    problem = core_inputs.least_squares(n=n, rows=case["rows"], d=d, seed=seed, device="cuda")
    state = {"kind": case["kind"], "core": binding.Core(GENERATOR_SEED, d, m),
             "ls": binding.LeastSquares(problem.A, problem.b),
             "x": core_inputs.gradients(1, d, seed=seed + 1_000_003, device="cuda")[0].contiguous()}
    state["core"].core_reserve_workspace(n, binding.CORE_F32)
    # the spectrum k^-1.5 / d has its largest eigenvalue at 1 / d: steps of a fraction of 1 / L
    state["h"] = (0.1 if case["kind"] == "agd" else 0.5) * d
    if case["kind"] == "agd":
        state["x_prev"] = state["x"].clone()
    elif case["kind"] == "guarded":
        state["f"] = state["core"].core_ls_loss(state["ls"], state["x"])
        state["accepted"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif case["kind"] == "decentralized":
        state["W"] = torch.from_numpy(core_inputs.gossip_matrix("ring", n)).to(torch.float32).cuda()
        state["rounds"] = case["rounds"]
        state["spread"] = torch.empty(1, dtype=torch.float32, device="cuda")
    return state


def prepare(case, seed):
    return _prepare_round(case, seed) if case["kind"] in ROUND_KINDS else _prepare_ls(case, seed)


def run(state):
    kind, core = state["kind"], state["core"]
    if kind == "round":
        return core.core_round(state["G"], state["pbar"], state["gtilde"])
    if kind == "host":
        return core.core_round_host(state["G"], state["pbar"], state["gtilde"])
    if kind == "machine":
        P = core.core_project(state["G"], state["P"])
        pbar = core.core_aggregate(state["P_all"], state["pbar"])
        return P, pbar, core.core_reconstruct(pbar, state["gtilde"])
    ls, x, h = state["ls"], state["x"], state["h"]
    if kind == "gd":
        return core.core_gd_step(ls, h, x)
    if kind == "agd":
        return core.core_agd_step(ls, h, 0.5, x, state["x_prev"])
    if kind == "guarded":
        core.core_gd_step_guarded(ls, h, x, state["f"], state["accepted"])
        return x, state["f"], state["accepted"]
    core.core_decentralized_step(ls, state["W"], state["rounds"], h, x, spread_dev=state["spread"])
    return x, state["spread"]


def work(case):
    kind, n, d, m = case["kind"], case["n"], case["d"], case["m"]
    if kind in ROUND_KINDS:
        size = 2 if case["dtype"] == "bf16" else 4
        rows = 1 if kind == "machine" else n
        # the gradients once, the estimate once, the messages; n + 1 multiply-adds per Gaussian.  The d m
        # Gaussians themselves (4 wide integer multiplies each, made once per direction) are in neither
        # figure and are what bounds all but the shortest vectors.
        small = 4 * m + (4 * m * (n + 1) if kind == "machine" else 0)
        return {"bytes": size * rows * d + 4 * d + small, "flops": 2 * (rows + 1) * d * m}
    # data matrices once (twice where f is evaluated at the trial point too), x read and written; residual,
    # gradient and round
    passes = 2 if kind == "guarded" else 1
    data = n * case["rows"] * d
    vectors = 4 if kind == "agd" else 2
    flops = (4 + 2 * (passes - 1)) * data + 2 * (n + 1) * d * m
    return {"bytes": 4 * (passes * (data + n * case["rows"]) + vectors * d), "flops": flops}


def tolerance(case):
    # fp32 sums of up to 1e9 products, and Gaussians that are right to 1e-6
    if case["kind"] in ROUND_KINDS:
        return {"rel": 2e-5}
    # x itself moves by a fraction of its size, through fp32 residuals and gradients; the spread is a maximum
    # of differences of messages that gossip has brought together
    return {"rel": 5e-5 if case["kind"] == "decentralized" else 2e-5}

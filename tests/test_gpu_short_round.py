"""Short vectors, whose round is one launch: a cluster keeps the Gaussians between projection and reconstruction.  At the sizes where it can
go wrong: CTAs without blocks, every cluster size, several machines' messages (the very numbers of the separate kernels), ragged
and unaligned rows, both sides of the lines to the separate kernels (which case takes which is asserted in test_short_plan.py), replays from
a graph, steps side by side.  Also rows a little too long for that, and the separate kernels at the sizes of the short ones."""
import threading

import numpy as np
import pytest
import torch

import core_inputs
import oracle
import test_gpu_round_paths as round_paths
from helpers import P_TOL, REC_TOL, rel_l2, row_norms
from test_short_plan import ROUTES, ROW_ROUTES

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def core_mod():
    import paper_2309_13307_b200 as core_mod
    core_mod.lib()
    return core_mod


@pytest.mark.parametrize("n,d,m,dtype,offset,pad", [
    (1, 1, 1, "f32", 0, 0), (1, 3, 4096, "bf16", 1, 0), (2, 4, 4097, "f32", 0, 0), (3, 33, 65, "f32", 1, 2), (4, 130, 16, "bf16", 0, 2),
    (5, 515, 33, "f32", 3, 0), (16, 257, 31, "bf16", 1, 0), (16, 1001, 40, "f32", 0, 3), (17, 300, 20, "f32", 0, 0), (1, 36, 300, "f32", 0, 0),
    (1, 7001, 37, "f32", 0, 0), (1, 65_533, 4, "bf16", 1, 0), (1, 65_537, 4, "f32", 0, 0), (4, 49_152, 4, "f32", 0, 0), (4, 49_157, 4, "f32", 0, 0),
    (2, 29, 3000, "f32", 0, 0), (8, 1500, 20, "bf16", 0, 0), (7, 260, 100, "f32", 0, 0), (6, 5000, 9, "f32", 0, 1), (2, 24_000, 6, "bf16", 0, 0),
])
def test_round_equals_its_parts_and_the_oracle(core_mod, n, d, m, dtype, offset, pad):
    from paper_2309_13307_b200 import binding
    G = core_inputs.gradients(n, d + offset, seed=d + m, dist="scaled_normal", dtype=dtype, device="cuda", ld=d + offset + pad)[:, offset:]
    Gh = core_inputs.to_oracle_array(G)
    ctx = core_mod.Core(5, d, m)
    ctx.core_set_round(2)
    P = ctx.core_project(G)
    pbar = ctx.core_aggregate(P)
    gt = ctx.core_reconstruct(pbar)
    Po, pbaro, gto = oracle.core_round(5, 2, m, Gh)
    assert (np.abs(P.cpu().numpy() - Po) <= P_TOL * row_norms(Gh)[:, None]).all()
    assert rel_l2(gt.cpu().numpy(), gto) <= REC_TOL
    pbar2, gt2 = ctx.core_round(G)
    assert torch.equal(pbar2, pbar) and torch.equal(gt2, gt)
    store = torch.full((d + 1,), 7.0, device="cuda")            # an estimate that does not start on 16 bytes
    ctx.core_set_round(2)
    assert torch.equal(ctx.core_reconstruct(pbar, store[1:]), gt) and store[0].item() == 7.0
    if n <= 16:
        P3 = torch.empty_like(P)
        binding.core_project_static(5, 2, m, G, P3)
        assert torch.equal(P3, P)


@pytest.fixture
def without_short_kernels(core_mod):
    from paper_2309_13307_b200 import binding
    binding.core_debug_short_kernels(False)
    yield
    binding.core_debug_short_kernels(True)


@pytest.mark.parametrize("n,d,m,dtype,offset,pad,ctas", ROUTES)
def test_routes(core_mod, n, d, m, dtype, offset, pad, ctas):
    from paper_2309_13307_b200 import binding
    test_round_equals_its_parts_and_the_oracle(core_mod, n, d, m, dtype, offset, pad)
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("routes of another device")
    G = core_inputs.gradients(n, d + offset, seed=1, dtype=dtype, device="cuda", ld=d + offset + pad)[:, offset:]
    ctx = core_mod.Core(5, d, m)
    pbar, gt = ctx.core_round(G)
    binding.core_debug_short_kernels(False)
    try:
        ctx.core_set_round(0)
        want, want_gt = ctx.core_round(G)
    finally:
        binding.core_debug_short_kernels(True)
    # messages kept apart are the same numbers by either; a single one is added up in another order, and so is the estimate
    if n > 1:
        assert torch.equal(pbar, want)
    assert float((pbar - want).abs().max()) <= P_TOL * float(G.float().norm(dim=1).mean())
    assert rel_l2(gt.cpu().numpy(), want_gt.cpu().numpy()) <= REC_TOL


@pytest.mark.parametrize("rows,d,m,ctas", ROW_ROUTES)
def test_sums_of_rows(core_mod, rows, d, m, ctas):
    G = core_inputs.gradients(rows, d, seed=d + m, device="cuda", ld=(d + 3) // 4 * 4)
    ctx = core_mod.Core(3, d, m)
    pbar, gt = ctx.core_debug_combined_round(G, 0.5)
    row = np.ascontiguousarray((0.5 * G.cpu().numpy().astype(np.float64).sum(axis=0, keepdims=True)).astype(np.float32))
    assert np.abs(pbar.cpu().numpy() - oracle.project(3, 0, m, row)[0]).max() <= P_TOL * row_norms(row)[0]
    assert rel_l2(gt.cpu().numpy(), oracle.reconstruct(3, 0, pbar.cpu().numpy().astype(np.float64), d)) <= REC_TOL


SINGLE_ROWS = round_paths.test_single_machine_projection.pytestmark[0].args[1]
RECONSTRUCTIONS = round_paths.test_short_reconstructions.pytestmark[0].args[1]


@pytest.mark.parametrize("d,m,dtype,offset", [*SINGLE_ROWS, *((d, m, t, o) for d in (1, 3, 5, 17) for m, t, o in ((4097, "f32", 1), (2, "bf16", 1), (9, "f32", 2),
                                                                                                               (21, "bf16", 6), (5000, "f32", 3)))])
def test_single_rows_without_the_short_kernels(core_mod, without_short_kernels, d, m, dtype, offset):
    round_paths.test_single_machine_projection(core_mod, d, m, dtype, offset)


@pytest.mark.parametrize("d,m", RECONSTRUCTIONS)
def test_reconstructions_without_the_short_kernels(core_mod, without_short_kernels, d, m):
    round_paths.test_short_reconstructions(core_mod, d, m)


@pytest.mark.parametrize("m,d", [(64, 2900), (3, 64_000), (400, 262_144), (100, 1_000_003)])
def test_rounding_errors_of_a_message(core_mod, m, d):
    """A chain of k additions of terms alike has an rms error of 2^-24 sqrt(k / 6) of the row's norm; with k <= 32 (24 in one launch) and the
    Gaussians' own errors (7.5e-8 each) and the later sums, 1.3e-7 together, that is 1.9e-7.  Chains of 64 would be 2.3e-7."""
    errors = []
    for seed in range(max(1, 400 // m)):
        G = core_inputs.gradients(1, d, seed=seed, device="cuda")
        Gh = core_inputs.to_oracle_array(G)
        got = core_mod.Core(100 + seed, d, m).core_project(G).cpu().numpy().astype(np.float64)
        errors.append((got - oracle.project(100 + seed, 0, m, Gh)) / row_norms(Gh)[0])
    assert np.sqrt(np.mean(np.square(errors))) <= 2.1e-7


@pytest.mark.parametrize("d,m", [(54, 16), (7, 3), (784, 64), (1000, 64), (1030, 64), (2900, 64)])
def test_order_of_a_single_message(core_mod, d, m):
    """The very numbers: up to four blocks of a lane in one chain, more in four sums; lanes in pairs, CTAs in ascending order."""
    from paper_2309_13307_b200 import binding
    plan = binding.core_debug_short_plan(m, d)
    per, lanes, blocks = plan["per"], plan["lanes"], (d + 3) // 4
    G = core_inputs.gradients(1, d, seed=m, device="cuda")
    ctx = core_mod.Core(8, d, m)
    got = ctx.core_project(G)[0].cpu().numpy()
    g = np.zeros(4 * blocks, np.float32)
    g[:d] = G[0].cpu().numpy()
    g = g.reshape(blocks, 4)
    z = np.stack([ctx.core_debug_gaussians(j, 0, blocks).cpu().numpy() for j in range(m)])

    def fma(a, b, c):                                              # the product is exact in 64 bits
        return (np.float64(a) * b.astype(np.float64) + c).astype(np.float32)

    want = np.zeros(m, np.float32)
    for first in range(0, blocks, per):
        end = min(first + per, blocks)
        parts = np.zeros((lanes, m), np.float32)
        for lane in range(lanes):
            s = np.zeros((4, m), np.float32)
            chain = 0 if per <= 4 * lanes else None
            for q in range(first + lane, end, lanes):
                for c in range(4):
                    to = c if chain is None else chain
                    s[to] = fma(g[q, c], z[:, q, c], s[to])
            parts[lane] = s[0] if chain == 0 else (s[0] + s[1]) + (s[2] + s[3])
        while len(parts) > 1:
            parts = parts[:len(parts) // 2] + parts[len(parts) // 2:]
        want = want + parts[0]
    assert np.array_equal(got, want)


STEPS = [(1, 5, 3, 8), (3, 40, 54, 16), (2, 7, 130, 9), (20, 11, 784, 64), (2, 150, 1201, 33), (3, 60, 1700, 100),   # one cluster
         (2, 30, 9000, 65), (1, 149, 4099, 256), (4, 20, 20_003, 20), (2, 9, 32_768, 256), (3, 70, 9578, 18)]          # separate kernels


@pytest.mark.parametrize("n,rows,d,m", STEPS)
def test_steps(core_mod, n, rows, d, m):
    problem = core_inputs.least_squares(n=n, rows=rows, d=d, seed=n + d, decay=0.5, device="cuda")
    Ah, bh = problem.A.cpu().numpy(), problem.b.cpu().numpy()
    ctx, ls = core_mod.Core(4, d, m), core_mod.LeastSquares(problem.A, problem.b)
    for offset in (0, 1):                                          # iterates that start on 16 bytes, and others
        x = core_inputs.gradients(1, d + offset, seed=1, device="cuda")[0][offset:]
        x_prev = core_inputs.gradients(1, d + offset, seed=2, device="cuda")[0][offset:]
        xo, xpo = x.cpu().numpy().astype(np.float64), x_prev.cpu().numpy().astype(np.float64)
        ctx.core_set_round(3)
        for t in (3, 4):
            ctx.core_agd_step(ls, 0.4, 0.7, x, x_prev)
            xo, xpo = oracle.agd_step(4, t, m, Ah, bh, 0.4, 0.7, xo, xpo)
        assert rel_l2(x.cpu().numpy(), xo) <= 1e-5 and rel_l2(x_prev.cpu().numpy(), xpo) <= 1e-5
    assert core_mod.core_device_status() == 0


@pytest.mark.parametrize("n,rows,d,m", [(20, 11, 784, 64), (2, 30, 9000, 65)])
def test_steps_replayed_from_a_graph_and_side_by_side(core_mod, n, rows, d, m):
    problem = core_inputs.least_squares(n=n, rows=rows, d=d, seed=7, decay=0.5, device="cuda")
    start = core_inputs.gradients(1, d, seed=1, device="cuda")[0].contiguous()

    def steps(stream, count, x):
        ctx, ls = core_mod.Core(4, d, m, stream=stream), core_mod.LeastSquares(problem.A, problem.b)
        for _ in range(count):
            ctx.core_gd_step(ls, 0.3, x)
        stream.synchronize()
        return ctx, ls

    want = start.clone()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx, ls = steps(stream, 6, want)
    # three steps of one graph, replayed twice from the same start: the same rounds, with nothing left over from the first
    x = start.clone()
    once = start.clone()
    steps(stream, 3, once)
    ctx.core_set_round(0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for _ in range(3):
            ctx.core_gd_step(ls, 0.3, x)
    for _ in range(2):
        x.copy_(start)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, once)
    del graph
    # three threads, a context and a stream each
    got = [start.clone() for _ in range(3)]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=steps, args=(torch.cuda.Stream(), 6, g)) for g in got]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert all(torch.equal(g, want) for g in got)
    assert core_mod.core_device_status() == 0


@pytest.mark.parametrize("d,m,dtype,offset", [(8192, 64, "f32", 0), (30_000, 64, "bf16", 0), (9001, 260, "f32", 1), (70_001, 33, "bf16", 3),
                                              (4097, 130, "f32", 0), (12_001, 100, "f32", 2), (50_000, 24, "f32", 0)])
def test_short_rows_of_many_ctas(core_mod, d, m, dtype, offset):
    """Rows a little too long for one launch: a column of partial sums per CTA, all CTAs resident together."""
    from paper_2309_13307_b200 import binding
    sm_count = torch.cuda.get_device_properties(0).multi_processor_count
    plan = binding.core_debug_row_plan(m, d, dtype=binding.CORE_BF16 if dtype == "bf16" else binding.CORE_F32, sm_count=sm_count)
    assert plan["grid_x"] == plan["tiles"] and not plan["turn"]
    G = core_inputs.gradients(1, d + offset, seed=d + m, dtype=dtype, device="cuda")[:, offset:]
    Gh = core_inputs.to_oracle_array(G)
    ctx = core_mod.Core(6, d, m)
    ctx.core_set_round(1)
    P = ctx.core_project(G)
    assert np.abs(P.cpu().numpy() - oracle.project(6, 1, m, Gh)).max() <= P_TOL * row_norms(Gh)[0]
    gt = ctx.core_reconstruct(P[0].contiguous())
    pbar2, gt2 = ctx.core_round(G)
    assert torch.equal(pbar2, P[0]) and torch.equal(gt2, gt)

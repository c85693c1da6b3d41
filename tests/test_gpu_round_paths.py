"""The round's special paths at the sizes where they can go wrong: one combined gradient row (any alignment, tile and
segment edges, staged by two warps or by all), reconstructions of short vectors shared out over warps and clusters, the
gossip rounds of a step in one launch, host rounds of one and of many slabs."""
import numpy as np
import pytest
import torch

import core_inputs
import oracle
from helpers import P_TOL, REC_TOL, rel_l2, row_norms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def core_mod():
    import paper_2309_13307_b200 as core_mod
    core_mod.lib()
    return core_mod


@pytest.mark.parametrize("d,m,dtype,offset", [
    (1, 1, "f32", 0), (3, 5, "f32", 1), (4, 4, "bf16", 0), (5, 1025, "f32", 3), (129, 20, "f32", 2), (257, 100, "bf16", 7),
    (1023, 7, "f32", 1), (4096, 3, "bf16", 5), (4097, 130, "f32", 0), (9001, 260, "bf16", 3), (20011, 17, "f32", 3),
])
def test_single_machine_projection(core_mod, d, m, dtype, offset):
    G = core_inputs.gradients(1, d + offset, seed=d + m, dtype=dtype, device="cuda")[:, offset:]
    ctx = core_mod.Core(7, d, m)
    ctx.core_set_round(3)
    Gh = core_inputs.to_oracle_array(G)
    want = oracle.project(7, 3, m, Gh)
    assert np.abs(ctx.core_project(G).cpu().numpy() - want).max() <= P_TOL * row_norms(Gh)[0]


@pytest.mark.parametrize("n,d,m,dtype,offset,pad", [
    (3, 400_003, 100, "f32", 1, 0), (2, 5_000_001, 8, "f32", 0, 0), (7, 1_048_577, 33, "bf16", 0, 3), (40, 262_145, 130, "f32", 0, 0),
    (5, 4_200_001, 8, "bf16", 3, 2), (2, 65_537, 520, "f32", 0, 7), (33, 2_100_000, 17, "bf16", 0, 0), (9, 33_000, 1030, "f32", 2, 1),
])
def test_round_on_the_mean_gradient_matches_its_messages(core_mod, n, d, m, dtype, offset, pad):
    """From 2^25 Gaussians on a round projects the mean gradient; the separate entry points form every message."""
    assert d * m >= 1 << 25
    G = core_inputs.gradients(n, d + offset, seed=n + m, dist="scaled_normal", dtype=dtype, device="cuda", ld=d + offset + pad)[:, offset:]
    ctx = core_mod.Core(2, d, m)
    pbar, gt = ctx.core_round(G)
    ctx.core_set_round(0)
    want = ctx.core_aggregate(ctx.core_project(G))
    scale = float(torch.linalg.vector_norm(G.float()) / n)
    assert float((pbar - want).abs().max()) <= 1e-5 * scale
    assert rel_l2(gt.cpu().numpy(), ctx.core_reconstruct(want).cpu().numpy()) <= 1e-4


@pytest.mark.parametrize("d,m", [(1, 1), (7, 33), (130, 2049), (800, 940), (3210, 3000), (33, 128), (4097, 515), (70_001, 65), (300_001, 17),
                                 (129, 64), (1000, 193)])
def test_short_reconstructions(core_mod, d, m):
    pbar = core_inputs.gradients(1, m, seed=d).numpy()[0]
    ctx = core_mod.Core(5, d, m)
    ctx.core_set_round(2)
    gt = ctx.core_reconstruct(torch.from_numpy(pbar).cuda())
    assert rel_l2(gt.cpu().numpy(), oracle.reconstruct(5, 2, pbar.astype(np.float64), d)) <= REC_TOL


@pytest.mark.parametrize("n,m,rounds", [(1, 9, 3), (3, 8, 1), (5, 17, 7), (32, 33, 4), (33, 5, 5), (128, 9, 2), (129, 6, 3)])
def test_gossip_rounds_of_a_step(core_mod, n, m, rounds):
    rows, d = 3, 40
    problem = core_inputs.least_squares(n=n, rows=rows, d=d, seed=n, decay=0.5, device="cuda")
    W = core_inputs.gossip_matrix("ring", n).astype(np.float32)
    ctx, ls = core_mod.Core(4, d, m), core_mod.LeastSquares(problem.A, problem.b)
    x = core_inputs.gradients(1, d, seed=1, device="cuda")[0].contiguous()
    spread = torch.zeros(1, dtype=torch.float32, device="cuda")
    xo, spread_o = oracle.decentralized_step(4, 0, m, problem.A.cpu().numpy(), problem.b.cpu().numpy(), W.astype(np.float64), rounds, 0.5,
                                             x.cpu().numpy().astype(np.float64), reader=n // 2)
    ctx.core_decentralized_step(ls, torch.from_numpy(W).cuda(), rounds, 0.5, x, reader=n // 2, spread_dev=spread)
    assert rel_l2(x.cpu().numpy(), xo) <= 1e-5
    assert abs(spread.item() - spread_o) <= 1e-4 * max(1.0, spread_o)


@pytest.mark.parametrize("n,d,m,dtype,pad", [(1, 5, 3, "f32", 0), (3, 4096, 9, "bf16", 0), (2, 4097, 8, "f32", 5), (5, 700_001, 12, "f32", 0),
                                             (17, 900_001, 5, "bf16", 3)])
def test_host_rounds(core_mod, n, d, m, dtype, pad):
    G = core_inputs.gradients(n, d, seed=n, dtype=dtype, ld=d + pad)
    ctx = core_mod.Core(6, d, m)
    pbar, gt = torch.empty(m), torch.empty(d)
    ctx.core_round_host(G, pbar, gt)
    ctx.core_set_round(0)
    pbar_d, gt_d = ctx.core_round(G.cuda())
    scale = float(torch.linalg.vector_norm(G.float()) / n)
    assert float((pbar - pbar_d.cpu()).abs().max()) <= 1e-5 * scale
    assert rel_l2(gt.numpy(), gt_d.cpu().numpy()) <= 1e-4

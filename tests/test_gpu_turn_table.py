"""The kernels that take the angles from a table: the Gaussians they use, the reconstruction's line of (unit, vector) pairs over
the warps, and the single-row projection's tiles, at sizes around the edges of units, warps, tables and CTA rows."""
import numpy as np
import pytest
import torch

import core_inputs
import oracle
from helpers import P_TOL, REC_TOL, rel_l2, row_norms

pytestmark = pytest.mark.gpu

XI_TOL = 4e-6       # |xi_gpu - xi_oracle|, element by element


@pytest.fixture(scope="module")
def core_mod():
    import paper_2309_13307_b200 as core_mod
    core_mod.lib()
    return core_mod


def windows(d, width=4096):
    """First, middle and last coordinates of a vector, starting on whole blocks."""
    middle, last = d // 2 // 4 * 4, max(0, d - width) // 4 * 4
    return [(0, min(width, d)), (middle, min(middle + width, d)), (last, d)]


@pytest.mark.parametrize("d,m,j", [(3_000_001, 9, 4), (94_720, 178, 0), (1_000_003, 100, 99)])
def test_gaussians(core_mod, d, m, j):
    """A message of one entry m reconstructs the vector of that entry itself; 3e6 coordinates hold radii down to 1e-3 and
    up to 5.6 and every entry of the table some hundred times."""
    pbar = torch.zeros(m, dtype=torch.float32, device="cuda")
    pbar[j] = m
    ctx = core_mod.Core(11, d, m)
    ctx.core_set_round(6)
    got = ctx.core_reconstruct(pbar).cpu().numpy().astype(np.float64)
    want = oracle.xi_range(11, 6, j, 0, d)
    assert np.abs(got - want).max() <= XI_TOL


@pytest.mark.parametrize("n,d,m,dtype,offset", [(1, 800_003, 21, "f32", 0), (1, 200_001, 100, "bf16", 3), (1, 30_000, 2049, "f32", 1),
                                                (2, 600_001, 61, "bf16", 0), (4, 600_001, 61, "f32", 1)])
def test_unit_vectors_read_the_projections_gaussians_back(core_mod, n, d, m, dtype, offset):
    """The message of e_k is xi_j[k], element by element: every other term of the sum is an exact zero."""
    from paper_2309_13307_b200 import binding
    size = 2 if dtype == "bf16" else 4
    G = torch.zeros((n, d + offset), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")[:, offset:]
    plan = binding.core_debug_row_plan(m, d, rows=n, ldg=d + offset, dtype=binding.CORE_BF16 if dtype == "bf16" else binding.CORE_F32,
                                       misaligned=offset * size % 16)
    assert plan["turn"]
    tile = 4 * plan["tile_q"]
    ctx = core_mod.Core(6, d, m)
    for k in sorted({0, 5, tile - 1, tile, d // 2, (plan["tiles"] - 1) * tile - 2, (plan["tiles"] - 1) * tile, d - 1}):
        G[:, k] = 1
        ctx.core_set_round(3)
        got = (ctx.core_project(G)[0] if n == 1 else ctx.core_round(G)[0]).cpu().numpy().astype(np.float64)
        G[:, k] = 0
        want = np.array([oracle.xi_range(6, 3, j, k, k + 1)[0] for j in range(m)])
        assert np.abs(got - want).max() <= XI_TOL, k


@pytest.mark.parametrize("d,m", [
    (94_717, 178), (94_720, 1025), (94_721, 2049), (151_552, 111), (151_553, 112), (303_100, 64), (1_000_003, 17), (6_000_000, 3),
    (17_000_001, 1), (17_000_001, 2), (100_003, 8192), (100_003, 8195), (700_001, 131),
])
def test_long_reconstructions(core_mod, d, m):
    pbar = core_inputs.gradients(1, m, seed=d % 1000 + m).numpy()[0]
    ctx = core_mod.Core(5, d, m)
    ctx.core_set_round(2)
    gt = ctx.core_reconstruct(torch.from_numpy(pbar).cuda()).cpu().numpy()
    for k0, k1 in windows(d, 4096 if m < 1000 else 640):
        assert rel_l2(gt[k0:k1], oracle.reconstruct_slice(5, 2, pbar.astype(np.float64), k0, k1)) <= REC_TOL


@pytest.mark.parametrize("d,m,kernel", [(2_422_789, 1, "wide"), (2_422_789, 5, "wide"), (2_424_833, 2, "wide"), (2_422_784, 3, "short"),
                                        (5_000_003, 3, "wide"), (9_786_709, 6, "turn"), (2_424_833, 8_193, "wide")])
def test_long_reconstructions_without_the_table(core_mod, d, m, kernel):
    from paper_2309_13307_b200 import binding
    assert binding.core_debug_reconstruct_plan(d, m)[0] == kernel
    test_long_reconstructions(core_mod, d, m)


@pytest.mark.parametrize("n,d,m", [(1, 4_000_003, 1), (3, 4_000_003, 2), (2, 2_500_001, 4), (1, 300_001, 1), (2, 1_000_003, 2)])
def test_rounds_of_few_vectors_equal_their_parts(core_mod, n, d, m):
    G = core_inputs.gradients(n, d, seed=m, device="cuda")
    ctx = core_mod.Core(5, d, m)
    pbar, gt = ctx.core_round(G)
    ctx.core_set_round(0)
    want = ctx.core_aggregate(ctx.core_project(G))
    assert float((pbar - want).abs().max()) <= P_TOL * float(G.norm(dim=1).mean())
    assert torch.equal(ctx.core_reconstruct(pbar), gt)


def test_reconstructions_do_not_depend_on_what_ran_before(core_mod):
    """Warps that share a unit meet in shared memory: the same bits on every launch."""
    d, m = 151_600, 333
    pbar = core_inputs.gradients(1, m, seed=1, device="cuda")[0]
    ctx = core_mod.Core(5, d, m)
    first = ctx.core_reconstruct(pbar).clone()
    for _ in range(20):
        assert torch.equal(ctx.core_reconstruct(pbar), first)


@pytest.mark.parametrize("n,d,m,dtype,offset,pad", [
    (1, 16_385, 1024, "f32", 0, 0), (1, 16_400, 1030, "bf16", 0, 8), (1, 5_600, 3073, "f32", 3, 0),
    (1, 49_153, 1024, "f32", 0, 0), (1, 48_900, 1030, "bf16", 0, 8), (1, 16_385, 3073, "f32", 3, 0), (1, 100_003, 170, "bf16", 5, 0),
    (1, 1_200_001, 14, "f32", 0, 0), (3, 600_001, 61, "f32", 0, 3), (4, 262_147, 130, "bf16", 1, 6), (20, 335_546, 101, "f32", 0, 2),
])
def test_projections(core_mod, n, d, m, dtype, offset, pad):
    """One row through core_project, several through the mean gradient of a round."""
    G = core_inputs.gradients(n, d + offset, seed=d + m, dtype=dtype, device="cuda", ld=d + offset + pad)[:, offset:]
    ctx = core_mod.Core(7, d, m)
    ctx.core_set_round(3)
    mean = G.float().cpu().numpy().astype(np.float64).mean(axis=0, keepdims=True)
    if n == 1:
        got = ctx.core_project(G).cpu().numpy()[0]
    else:
        got = ctx.core_round(G)[0].cpu().numpy()
    want = oracle.project(7, 3, m, np.ascontiguousarray(mean.astype(np.float32)))[0]
    # fp32 rounding of the mean itself: 2^-24 of its norm at most, four decimal digits below the bar
    assert np.abs(got - want).max() <= P_TOL * row_norms(mean.astype(np.float32))[0]


@pytest.mark.parametrize("n,d,m", [(2, 1_130_988, 18), (2, 1_090_804, 17), (2, 1_136_948, 24), (1, 1_138_688, 32), (2, 2_324_170, 34),
                                   (1, 1_175_641, 45), (1, 1_174_605, 48), (2, 1_174_604, 48)])
def test_projections_with_the_longest_tiles(core_mod, n, d, m):
    """Tiles close to the longest of 2048 blocks: beside the table of angles they take most of a CTA's shared memory."""
    from paper_2309_13307_b200 import binding
    G = core_inputs.gradients(n, d, seed=d + m, device="cuda", ld=(d + 3) // 4 * 4)
    plan = binding.core_debug_row_plan(m, d, rows=n, ldg=G.stride(0))
    assert plan["turn"] and plan["tile_q"] > 1968
    ctx = core_mod.Core(7, d, m)
    ctx.core_set_round(3)
    mean = np.ascontiguousarray(G.cpu().numpy().astype(np.float64).mean(axis=0, keepdims=True).astype(np.float32))
    want = oracle.project(7, 3, m, mean)[0]
    got = [ctx.core_round(G)[0]]
    if n == 1:
        ctx.core_set_round(3)
        P = torch.empty((1, m), dtype=torch.float32, device="cuda")
        binding.core_project_static(7, 3, m, G, P)
        got += [ctx.core_project(G)[0], P[0]]
    for p in got:
        assert np.abs(p.cpu().numpy() - want).max() <= P_TOL * row_norms(mean)[0]
        assert torch.equal(p, got[0])


@pytest.mark.parametrize("n,d,m", [(1, 2_200_673, 45), (2, 3_801_345, 20)])
def test_host_rounds_with_the_longest_tiles(core_mod, n, d, m):
    from paper_2309_13307_b200 import binding
    plans = [binding.core_debug_row_plan(m, s, rows=n, ldg=(s + 7) // 8 * 8) for s in binding.core_debug_host_slabs(d, n)]
    assert any(p["turn"] and p["tile_q"] > 1968 for p in plans)
    G = core_inputs.gradients(n, d, seed=d, device="cuda")
    ctx = core_mod.Core(7, d, m)
    pbar, gt = torch.empty(m, dtype=torch.float32), torch.empty(d, dtype=torch.float32)
    ctx.core_round_host(G.cpu(), pbar, gt)
    ctx.core_set_round(0)
    want, want_gt = ctx.core_round(G)
    # two orders of fp32 sums over the same Gaussians
    assert float((pbar - want.cpu()).norm()) <= 2e-5 * float(want.norm())
    assert rel_l2(gt.numpy(), want_gt.cpu().numpy()) <= 2e-5


@pytest.mark.parametrize("m", [2, 3, 7, 8, *range(12, 21)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_one_row_gives_the_same_bits_wherever_it_starts(core_mod, m, dtype):
    """Around the lines between the kernels for one row; ldg is the stride of rows that are not there."""
    from paper_2309_13307_b200 import binding
    d = (1 << 21) + 5
    row = core_inputs.gradients(1, d, seed=m, dtype=dtype, device="cuda")[0]
    store = torch.zeros(d + 16, dtype=row.dtype, device="cuda")
    ctx = core_mod.Core(7, d, m)
    P = torch.empty((1, m), dtype=torch.float32, device="cuda")
    want = ctx.core_project(row[None]).clone()
    for offset in range(8):
        store[offset:offset + d] = row
        for ldg in (d, d + 1, d + 3, d + 6):
            P.zero_()
            rc = binding.lib().core_project(ctx._h, store.data_ptr() + offset * store.element_size(),
                                            binding.CORE_BF16 if dtype == "bf16" else binding.CORE_F32, 1, ldg, P.data_ptr())
            assert rc == 0 and torch.equal(P, want), (offset, ldg)

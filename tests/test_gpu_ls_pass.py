"""The single pass over A (gradients, loss, the summed gradient of a step) at the sizes where it changes shape: one
column per lane up to a cluster of CTAs per row, rows per CTA from less than one batch on, machine boundaries inside a
CTA's range, rows of every alignment.  Bars as in the other least-squares tests: relative L2 <= 1e-5 against the oracle."""
import numpy as np
import pytest
import torch

import core_inputs
import oracle
from helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def core_mod():
    import paper_2309_13307_b200 as core_mod
    core_mod.lib()
    return core_mod


@pytest.mark.parametrize("n,rows,d,offset", [
    (1, 1, 1, 0), (3, 700, 1, 1), (2, 5, 31, 0), (50, 37, 54, 0), (7, 333, 64, 2), (64, 16, 65, 3),   # several rows at a time
    (2, 3000, 127, 1), (5, 61, 129, 0), (3, 200, 256, 0), (2, 999, 257, 3), (4, 77, 511, 1), (3, 65, 512, 0),  # one warp
    (6, 50, 513, 0), (8, 331, 600, 2), (2, 90, 768, 0), (2, 150, 769, 1), (9, 120, 784, 0), (2, 400, 1023, 2),  # per row
    (1, 150, 1024, 0), (2, 90, 1025, 0), (3, 50, 1536, 0),                                               # 2 warps
    (3, 50, 2047, 1), (3, 151, 2049, 0), (2, 47, 2561, 1), (3, 40, 3072, 0),                             # 4
    (2, 70, 3073, 0), (2, 149, 4096, 0), (1, 40, 4097, 1), (3, 60, 5500, 3), (2, 51, 6145, 1), (2, 80, 8192, 0),  # 8
    (1, 33, 8193, 3), (40, 9, 9001, 1), (5, 7, 12000, 0), (2, 75, 16384, 0),                             # 16
    (1, 80, 16385, 0), (3, 30, 20001, 1), (16, 5, 24000, 0), (1, 37, 33000, 2),                          # clusters of 2 and 4
])
def test_gradients_loss_and_step(core_mod, n, rows, d, offset):
    A = core_inputs.gradients(1, n * rows * d + offset, seed=n + rows + d, device="cuda")[0][offset:].view(n, rows, d)
    b = core_inputs.gradients(n, rows, seed=5, device="cuda").contiguous()
    x = core_inputs.gradients(1, d, seed=6, device="cuda")[0].contiguous()
    x_prev = core_inputs.gradients(1, d, seed=7, device="cuda")[0].contiguous()
    Ah, bh, xh = A.cpu().numpy(), b.cpu().numpy(), x.cpu().numpy().astype(np.float64)
    ctx, ls = core_mod.Core(3, d, 8), core_mod.LeastSquares(A, b)
    G = ctx.core_ls_gradients(ls, x).cpu().numpy()
    want = oracle.ls_grad(Ah, bh, xh)
    for i in range(n):
        assert rel_l2(G[i], want[i]) <= 1e-5, (i, rel_l2(G[i], want[i]))
    f0 = oracle.ls_loss(Ah, bh, xh)
    assert abs(float(ctx.core_ls_loss(ls, x).item()) - f0) <= 1e-5 * f0
    # a step's round on the summed gradient, at the look-ahead point of the accelerated step
    h, beta = 0.01, 0.3
    xa, xp = x.clone(), x_prev.clone()
    ctx.core_agd_step(ls, h, beta, xa, xp)
    want_x, want_p = oracle.agd_step(3, 0, 8, Ah, bh, h, beta, xh, x_prev.cpu().numpy().astype(np.float64))
    assert rel_l2(xa.cpu().numpy(), want_x) <= 1e-4 and np.array_equal(xp.cpu().numpy(), x.cpu().numpy())
    # the comparison step reads the rows backwards for the trial point's loss
    f = torch.tensor([f0], dtype=torch.float64, device="cuda")
    xg, h = x.clone(), 1e-6
    ctx.core_set_round(0)
    accepted = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.core_gd_step_guarded(ls, h, xg, f, accepted)
    trial = oracle.gd_step(3, 0, 8, Ah, bh, h, xh)
    f1 = oracle.ls_loss(Ah, bh, trial)
    if accepted.item():
        assert abs(f.item() - f1) <= 1e-5 * f1 and rel_l2(xg.cpu().numpy(), trial) <= 1e-5
    else:
        assert torch.equal(xg, x) and f.item() == f0 and f1 >= f0 * (1 - 1e-5)
    assert core_mod.core_device_status() == 0


@pytest.mark.parametrize("n,rows,d", [(1, 3, 1), (1, 147, 1), (7, 60, 1), (1, 443, 1), (3, 41, 2), (1, 295, 2), (1, 170, 3)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_rows_shorter_than_a_copy_unit(core_mod, n, rows, d, offset):
    """Rows of a few floats: the ends of the matrix lie within one 16-byte unit of CTAs that are not the first or the last."""
    A = core_inputs.gradients(1, n * rows * d + offset, seed=n + rows + d, device="cuda")[0][offset:].view(n, rows, d)
    b = core_inputs.gradients(n, rows, seed=5, device="cuda").contiguous()
    x = core_inputs.gradients(1, d, seed=6, device="cuda")[0].contiguous()
    Ah, bh, xh = A.cpu().numpy(), b.cpu().numpy(), x.cpu().numpy().astype(np.float64)
    ctx, ls = core_mod.Core(3, d, 8), core_mod.LeastSquares(A, b)
    G = ctx.core_ls_gradients(ls, x).cpu().numpy()
    want = oracle.ls_grad(Ah, bh, xh)
    # fp32 sums of `rows` products whose terms may cancel: relative to the sum of their magnitudes
    terms = np.abs(Ah.astype(np.float64)) * np.abs(np.einsum("nrd,d->nr", Ah.astype(np.float64), xh) - bh)[:, :, None]
    assert (np.abs(G - want) <= 1e-5 * terms.mean(axis=1) + 1e-12).all()
    f0 = oracle.ls_loss(Ah, bh, xh)
    assert abs(float(ctx.core_ls_loss(ls, x).item()) - f0) <= 1e-5 * f0
    assert core_mod.core_device_status() == 0


@pytest.mark.parametrize("n,rows,d,offset", [
    (2, 75, 10240, 0), (1, 40, 10241, 1), (2, 150, 12288, 0), (3, 50, 12289, 1), (1, 160, 13824, 0), (2, 30, 14064, 2), (2, 75, 14065, 3),   # a CTA
    (2, 40, 20480, 0), (1, 37, 20481, 1), (2, 37, 28126, 0), (1, 30, 28133, 3), (1, 20, 100003, 0),                                   # clusters
    (2, 1776, 12289, 1), (1, 3551, 14064, 0), (3, 197, 25505, 3), (1, 592, 28126, 0), (1, 120, 56001, 1), (1, 57, 110003, 0)])      # 28 columns: rows enough
def test_columns_per_lane_of_long_rows(core_mod, n, rows, d, offset):
    """20, 24, 28 and 32 columns per lane, two rows at a time or one, up to the last row length of each and on both sides of the number of
    rows from which 28 columns are taken."""
    test_gradients_loss_and_step(core_mod, n, rows, d, offset)

"""GPU parity of the machine gradients g_i = A_i^T (A_i x - b_i) / rows of the least-squares driver
(Algorithm 2's local computation) for both device paths: the single pass over A (rows of up to 131072
columns, x of any alignment) and the two passes over longer rows.  Bar: relative L2 <= 1e-5 per machine against the
fp64 oracle."""
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


@pytest.mark.parametrize("n,rows,d", [(1, 1, 4), (2, 7, 1024), (3, 50, 1028), (8, 300, 8192), (4, 33, 2052),
                                      (2, 5, 8196), (3, 20, 1001), (40, 9, 512)])
def test_gradients_both_paths(core_mod, n, rows, d):
    ls_in = core_inputs.least_squares(n=n, rows=rows, d=d, seed=n + rows, device="cuda")
    ls = core_mod.LeastSquares(ls_in.A, ls_in.b)
    ctx = core_mod.Core(1, d, 4)
    store = core_inputs.gradients(1, d + 4, seed=3, device="cuda")[0].contiguous()
    x_aligned = store[:d].clone()
    x_shifted = store[1:d + 1]                      # 4-byte offset
    Ah, bh = ls_in.A.cpu().numpy(), ls_in.b.cpu().numpy()
    for x in (x_aligned, x_shifted):
        G = ctx.core_ls_gradients(ls, x.contiguous() if x is x_aligned else x).cpu().numpy()
        Go = oracle.ls_grad(Ah, bh, x.cpu().numpy().astype(np.float64))
        for i in range(n):
            assert rel_l2(G[i], Go[i]) <= 1e-5, (i, rel_l2(G[i], Go[i]))
    # bitwise reproducible
    xs = x_aligned.clone()
    a = ctx.core_ls_gradients(ls, xs)
    b = ctx.core_ls_gradients(ls, xs)
    assert torch.equal(a, b)


@pytest.mark.parametrize("n,rows,d,offset", [(2, 5, 131073, 0), (1, 9, 131076, 1), (3, 4, 140000, 0)])
def test_rows_too_long_for_the_single_pass(core_mod, n, rows, d, offset):
    """Two passes over A: residuals, then A^T r; the steps and the loss on top of them."""
    from paper_2309_13307_b200 import binding
    assert binding.core_debug_ls_reads(n, rows, d, True, 0)[0] == 0                # the single pass does not apply
    A = core_inputs.gradients(1, n * rows * d + offset, seed=n + rows, device="cuda")[0][offset:].view(n, rows, d)
    b = core_inputs.gradients(n, rows, seed=5, device="cuda").contiguous()
    store = core_inputs.gradients(1, d + 1, seed=6, device="cuda")[0].contiguous()
    Ah, bh = A.cpu().numpy(), b.cpu().numpy()
    ctx, ls = core_mod.Core(3, d, 4), core_mod.LeastSquares(A, b)
    for x in (store[:d], store[1:]):                # aligned, and 4 bytes off
        xh = x.cpu().numpy().astype(np.float64)
        G = ctx.core_ls_gradients(ls, x).cpu().numpy()
        want = oracle.ls_grad(Ah, bh, xh)
        for i in range(n):
            assert rel_l2(G[i], want[i]) <= 1e-5, (i, rel_l2(G[i], want[i]))
        f = oracle.ls_loss(Ah, bh, xh)
        assert abs(float(ctx.core_ls_loss(ls, x).item()) - f) <= 1e-5 * f
    x, x_prev, h, beta = store[:d].clone(), store[1:].clone(), 1e-3, 0.3
    xh, ph = x.cpu().numpy().astype(np.float64), x_prev.cpu().numpy().astype(np.float64)
    ctx.core_agd_step(ls, h, beta, x, x_prev)
    want_x, want_p = oracle.agd_step(3, 0, 4, Ah, bh, h, beta, xh, ph)
    assert rel_l2(x.cpu().numpy(), want_x) <= 1e-4 and rel_l2(x_prev.cpu().numpy(), want_p) <= 1e-6
    x = store[:d].clone()
    ctx.core_set_round(0)
    ctx.core_gd_step(ls, h, x)
    assert rel_l2(x.cpu().numpy(), oracle.gd_step(3, 0, 4, Ah, bh, h, xh)) <= 1e-5

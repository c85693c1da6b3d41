"""A least-squares pass whose rows never arrive: the copy of one chunk is left out, the wait for it runs out after 100 ms,
the kernel ends by its normal exit with its other copies done, the status word tells, and nothing wrong passes for a result."""
import time

import pytest
import torch

import core_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def core_mod():
    import paper_2309_13307_b200 as core_mod
    core_mod.lib()
    return core_mod


# one warp per row with the held-back chunk among the first and behind the ring's, 2, 8 and 16 warps per row, clusters
@pytest.mark.parametrize("n,rows,d,chunk", [(2, 30000, 64, 0), (2, 30000, 64, 20), (4, 600, 600, 3), (3, 500, 5500, 1),
                                            (2, 400, 9001, 2), (8, 300, 16384, 9), (4, 150, 20001, 1), (1, 200, 33000, 0)])
def test_a_copy_that_never_arrives(core_mod, n, rows, d, chunk):
    A = core_inputs.gradients(n * rows, d, seed=d, device="cuda").view(n, rows, d)
    b = core_inputs.gradients(n, rows, seed=5, device="cuda").contiguous()
    x = core_inputs.gradients(1, d, seed=6, device="cuda")[0].contiguous()
    ctx, ls = core_mod.Core(3, d, 8), core_mod.LeastSquares(A, b)
    good_G, good_f = ctx.core_ls_gradients(ls, x), ctx.core_ls_loss(ls, x)
    good_x = x.clone()
    ctx.core_gd_step(ls, 0.01, good_x)
    assert core_mod.core_device_status() == 0 and bool(torch.isfinite(good_x).all())

    ls.core_debug_hold_back(chunk)
    t0 = time.perf_counter()
    G = ctx.core_ls_gradients(ls, x)
    # in a cluster one CTA waits for rows, the others for its share of their dot products; synchronises, reads and clears
    assert core_mod.core_device_status() == (22 if d > 16384 else 21)
    assert time.perf_counter() - t0 < 5.0
    assert bool(torch.isnan(G).any(dim=1).all())                       # every machine has rows that never arrived
    assert bool(torch.isnan(ctx.core_ls_loss(ls, x)).all())
    assert core_mod.core_device_status() in (21, 22)
    x1, x2, x2_prev, x3 = (x.clone() for _ in range(4))
    ctx.core_gd_step(ls, 0.01, x1)
    ctx.core_agd_step(ls, 0.01, 0.5, x2, x2_prev)
    assert bool(torch.isnan(x1).all()) and bool(torch.isnan(x2).all())
    f, taken = good_f.clone(), torch.full((1,), 7, dtype=torch.int32, device="cuda")
    ctx.core_gd_step_guarded(ls, 0.01, x3, f, taken)
    assert torch.equal(x3, x) and torch.equal(f, good_f) and int(taken) == 0
    assert core_mod.core_device_status() in (21, 22)

    # the device and the handle go on as before
    ls.core_debug_hold_back(-1)
    ctx.core_set_round(0)
    assert torch.equal(ctx.core_ls_gradients(ls, x), good_G) and torch.equal(ctx.core_ls_loss(ls, x), good_f)
    x4 = x.clone()
    ctx.core_gd_step(ls, 0.01, x4)
    assert torch.equal(x4, good_x) and core_mod.core_device_status() == 0

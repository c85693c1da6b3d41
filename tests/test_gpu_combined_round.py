"""The round that ends a least-squares step: one message of scale times the sum of the rows, by the single launch of short vectors and by the
separate kernels of longer ones, for one row as for many."""
import numpy as np
import pytest
import torch

import core_inputs
import oracle
from helpers import P_TOL, REC_TOL, rel_l2, row_norms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,d,m,pad", [(1, 1, 1, 0), (1, 1003, 16, 1), (1, 4096, 8, 0), (2, 600, 24, 3), (9, 2000, 9, 0), (30, 130, 64, 2),
                                          (150, 300, 5, 0), (150, 3000, 16, 4), (1, 30_001, 33, 0), (3, 9000, 64, 1), (150, 20_000, 20, 0)])
def test_scale_times_the_sum_of_the_rows(rows, d, m, pad):
    import paper_2309_13307_b200 as core_mod
    G = core_inputs.gradients(rows, d, seed=d + m, device="cuda", ld=d + pad)
    ctx = core_mod.Core(3, d, m)
    ctx.core_set_round(4)
    pbar, gt = ctx.core_debug_combined_round(G, 0.25)
    # the sum of up to 150 rows rounds to 150 * 2^-24 of its terms at most, a tenth of the bar
    row = np.ascontiguousarray((0.25 * G.cpu().numpy().astype(np.float64).sum(axis=0, keepdims=True)).astype(np.float32))
    assert np.abs(pbar.cpu().numpy() - oracle.project(3, 4, m, row)[0]).max() <= P_TOL * row_norms(row)[0]
    assert rel_l2(gt.cpu().numpy(), oracle.reconstruct(3, 4, pbar.cpu().numpy().astype(np.float64), d)) <= REC_TOL

"""core_project on both sides of the line between the scalar and the tensor-memory projection, element by element."""
import numpy as np
import pytest

import core_inputs
import oracle
from helpers import P_TOL, row_norms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(8, 65), (9, 64), (9, 65), (16, 127), (16, 129), (17, 33), (24, 64), (25, 32), (25, 33), (25, 64), (32, 40),
                                 (33, 65), (41, 191), (50, 33), (64, 64)])
@pytest.mark.parametrize("d,dtype", [(2_003, "f32"), (8_192, "bf16")])
def test_messages_on_both_sides_of_the_rule(n, m, d, dtype):
    import paper_2309_13307_b200 as core_mod
    G = core_inputs.gradients(n, d, seed=n * m, dtype=dtype, dist="scaled_normal", device="cuda")
    Gh = core_inputs.to_oracle_array(G)
    ctx = core_mod.Core(3, d, m)
    ctx.core_set_round(1)
    diff = np.abs(ctx.core_project(G).cpu().numpy() - oracle.project(3, 1, m, Gh))
    assert (diff <= P_TOL * np.asarray(row_norms(Gh))[:, None]).all()

"""Launch statistics of the 3D element multigrid: every kernel is booked.  One fine level above 15^3
takes two launches of layers (even, odd) and one of residual and restriction; the levels from
15^3 down take one."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m1,fine", [(15, 0), (31, 1), (63, 2)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_layers_are_counted(m1, fine, precision):
    from paper_2410_22686_gb300 import Solver
    a = np.exp(0.3 * S.random_vector((m1 + 2,) * 3, 4))
    sol = Solver(3, m1, 1, 1.0, 1e-3, 0.3, a, spatial="mg", precision=precision, max_iter=2, space="fe", tiles=None)
    v = torch.from_numpy(S.random_vector((2, 1) + (m1,) * 3, 9)).cuda()
    sol.stats_reset()
    sol.apply_precond(v)
    got = {k: s["launches"] for k, s in sol.stats().items()}
    sol.close()
    assert got["mg_smooth_rb"] == 2 * fine
    assert got["mg_resid_restrict"] == fine
    assert got["mg_coarse_cycle"] == 1

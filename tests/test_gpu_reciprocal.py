"""The FP64 reciprocal of the shifted diagonals (an FP32 seed and one cubic step inside the FP32
normal range, the division outside) in the multigrid apply: coefficients that keep |sigma + d|^2
inside that range, at its upper edge (2^123) and far above it."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import precond as opc, system as osy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e17, 3e17, 1e18, 1e30])
@pytest.mark.parametrize("d,m1,n", [(2, 31, 8), (2, 63, 4), (3, 7, 8)])
def test_fp64_apply_matches_oracle(d, m1, n, scale):
    from paper_2410_22686_gb300 import Solver
    a = scale * np.exp(0.5 * S.random_vector((m1 + 2,) * d, 7))
    gamma, eps = 1e-4, 0.25
    sol = Solver(d, m1, n, 1.0, gamma, eps, a, spatial="mg", max_iter=4, tiles=None)
    v = S.random_vector((2, n) + (m1,) * d, 8)
    w = sol.apply_precond(torch.from_numpy(v).cuda()).cpu().numpy()
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, gamma)
    ref = opc.apply_Peps_inv(v, n, alpha, eps, opc.MGSpatialSolver(a, tau))
    assert np.abs(w - ref).max() <= 1e-12 * np.abs(ref).max()
    sol.close()

"""FP32 applies at the paper's eps = tau / 2 (down to 5e-4; FP32 is taken automatically to 1e-4), against
the oracle: lengths by the direct sum, the chirp-z method and the register FFT.  The scalings
eps^{j/n} and their inverses carry the transforms' errors, sqrt(n) 2^-24 at most (n roundings of
random sign), to 1 / eps times that."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import precond as opc, system as osy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spatial", ["fst", "mg"])
@pytest.mark.parametrize("m1,n", [(15, 511), (12, 255), (7, 1023), (15, 512), (7, 100)])
def test_fp32_apply_matches_oracle(m1, n, spatial):
    from paper_2410_22686_gb300 import Solver
    if spatial == "mg" and (m1 & (m1 + 1)):
        pytest.skip("multigrid needs m1 = 2^k - 1")
    a = None if spatial == "fst" else np.exp(0.4 * S.random_vector((m1 + 2, m1 + 2), n))
    gamma, tau, alpha = 1e-4, osy.time_step(1.0, n), osy.alpha_weight(1.0, n, 1e-4)
    eps = 0.5 * tau
    sol = Solver(2, m1, n, 1.0, gamma, eps, a, spatial=spatial, precision="fp32", max_iter=2, tiles=None)
    v = S.random_vector((2, n, m1, m1), 17)
    w = sol.apply_precond(torch.from_numpy(v).cuda()).cpu().numpy()
    sol.close()
    ref = opc.apply_Peps_inv(v, n, alpha, eps, opc.make_spatial_solver(spatial, a, m1, 2, tau))
    assert np.abs(w - ref).max() <= np.sqrt(n) * 2.0 ** -24 / eps * np.abs(ref).max()

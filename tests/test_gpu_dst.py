"""Sine transforms of lines whose m + 1 is not a power of two (products with half of the DST-I
matrix), inside the preconditioner, against the oracle: FP64 1e-12, FP32 1e-5 (the
tolerances of the fast transforms; a line's sum of m/2 terms is shorter than the m of the
matrix product)."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import fe, precond as opc, system as osy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_22686_gb300 import build
    build.build()
    assert torch.cuda.is_available()


# even and odd m (with and without a middle point), one output a parity, one to four outputs a
# thread, tiles of one line (m = 1100 in FP64) up to 32, lines left over; m = 511 is the FP64
# length beyond the register FFTs
@pytest.mark.parametrize("space", ["fd", "fe"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("d,m1,n", [(2, 2, 3), (2, 4, 5), (2, 5, 300), (2, 12, 8), (2, 33, 40), (2, 100, 4),
                                    (2, 129, 2), (2, 511, 1), (2, 1100, 1), (3, 2, 4), (3, 6, 9), (3, 11, 64),
                                    (3, 20, 3)])
def test_apply_matches_oracle(d, m1, n, precision, tol, space):
    from paper_2410_22686_gb300 import Solver
    gamma, eps = 1e-4, 0.25
    sol = Solver(d, m1, n, 1.0, gamma, eps, None, spatial="fst", precision=precision, max_iter=2, space=space,
                 tiles=None)
    v = S.random_vector((2, n) + (m1,) * d, 17)
    w = sol.apply_precond(torch.from_numpy(v).cuda()).cpu().numpy()
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, gamma)
    spat = (fe.FSTSpatialSolverFE if space == "fe" else opc.FSTSpatialSolver)(m1, d, tau)
    ref = opc.apply_Peps_inv(v, n, alpha, eps, spat)
    assert np.abs(w - ref).max() / np.abs(ref).max() <= tol
    sol.close()

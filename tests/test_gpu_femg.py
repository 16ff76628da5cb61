"""The fused element multigrid kernels (a level's sweep, residual and restriction by strips
of rows; the small levels in one launch) inside the preconditioner, against the oracle's
level-by-level cycle: FP64 1e-12 and FP32 1e-5, the tolerances of the preconditioner
(tests/test_gpu_fe_var.py)."""
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


def _apply(d, m1, n, precision, a, v, gamma=1e-3, eps=0.3):
    from paper_2410_22686_gb300 import Solver
    sol = Solver(d, m1, n, 1.0, gamma, eps, a, spatial="mg", precision=precision, max_iter=2, space="fe", tiles=None)
    w = sol.apply_precond(torch.from_numpy(v).cuda())
    sol.close()
    return w


# strips of 4 rows with a remainder (few planes), of 8 and 16 (many planes); one fine level
# above the small ones (63 in FP64, 127 in FP32) and two (127, 255)
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("m1,n", [(63, 1), (63, 200), (127, 2), (127, 40), (255, 3)])
def test_strips_match_oracle(m1, n, precision, tol):
    a = np.exp(0.5 * S.random_vector((m1 + 2, m1 + 2), 3))
    v = S.random_vector((2, n, m1, m1), 4)
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, 1e-3)
    ref = opc.apply_Peps_inv(v, n, alpha, 0.3, fe.MGSpatialSolverFE(a, tau))
    w = _apply(2, m1, n, precision, a, v).cpu().numpy()
    assert np.abs(w - ref).max() / np.abs(ref).max() <= tol


def test_rows_too_wide_for_a_strip_agree_with_strips():
    # 2047 points a row: an FP32 strip fits, an FP64 one does not (per-level kernels there)
    m1, n = 2047, 1
    a = np.exp(0.3 * S.random_vector((m1 + 2, m1 + 2), 5))
    v = S.random_vector((2, n, m1, m1), 6)
    w32, w64 = (_apply(2, m1, n, p, a, v) for p in ("fp32", "fp64"))
    assert float((w32 - w64).abs().max() / w64.abs().max()) <= 1e-5


# 3D: the small levels alone (1, 7, 15), one fine level (31: two strips of coarse rows with a
# remainder), many planes
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("m1,n", [(1, 2), (7, 40), (15, 3), (31, 1), (31, 20)])
def test_layers_match_oracle(m1, n, precision, tol):
    a = np.exp(0.4 * S.random_vector((m1 + 2,) * 3, 7))
    v = S.random_vector((2, n) + (m1,) * 3, 8)
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, 1e-3)
    ref = opc.apply_Peps_inv(v, n, alpha, 0.3, fe.MGSpatialSolverFE(a, tau))
    w = _apply(3, m1, n, precision, a, v).cpu().numpy()
    assert np.abs(w - ref).max() / np.abs(ref).max() <= tol


def test_layers_of_several_strips_agree_between_precisions():
    # 63 rows a layer: strips of 16 row pairs in FP32 and 4 in FP64
    m1, n = 63, 3
    a = np.exp(0.4 * S.random_vector((m1 + 2,) * 3, 9))
    v = S.random_vector((2, n) + (m1,) * 3, 10)
    w32, w64 = (_apply(3, m1, n, p, a, v) for p in ("fp32", "fp64"))
    assert float((w32 - w64).abs().max() / w64.abs().max()) <= 1e-5

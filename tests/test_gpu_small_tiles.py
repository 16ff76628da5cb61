"""Time and sine transforms where the chip would be left idle by full CTAs: a quarter of the
columns or lines per CTA, against the oracle at sizes on both sides of the switch (two CTAs
an SM), with columns and lines left over, and the iterates' correction added at every
parity of a point.  FP64 1e-12, FP32 1e-5, BF16 storage 3e-2 (tests/test_gpu_parity.py)."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import precond as opc, system as osy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_22686_gb300 import build
    build.build()
    assert torch.cuda.is_available()


def _check(d, m1, n, spatial, precision, tol):
    from paper_2410_22686_gb300 import Solver
    a = None if spatial == "fst" else np.exp(0.4 * S.random_vector((m1 + 2,) * d, n))
    gamma, eps = 1e-4, 0.25
    sol = Solver(d, m1, n, 1.0, gamma, eps, a, spatial=spatial, precision=precision, max_iter=2, tiles=None)
    v = S.random_vector((2, n) + (m1,) * d, 17)
    w = sol.apply_precond(torch.from_numpy(v).cuda()).cpu().numpy()
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, gamma)
    ref = opc.apply_Peps_inv(v, n, alpha, eps, opc.make_spatial_solver(spatial, a, m1, d, tau))
    assert np.abs(w - ref).max() / np.abs(ref).max() <= tol
    sol.close()


# time transforms: n = 8 .. 256 with 304 CTAs of 256 threads as the line (63^2 and 127^2 columns
# lie on either side of it for n >= 32), n = 1024 always whole
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("m1,n", [(9, 8), (10, 16), (63, 32), (127, 32), (63, 64), (30, 128), (63, 256), (127, 16),
                                  (11, 1024)])
def test_time_transforms(m1, n, precision, tol):
    _check(2, m1, n, "fst", precision, tol)


# sine transforms of 7, 15, 31, 63, 127 points on few and on many planes, in 2D and 3D
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("d,m1,n", [(2, 7, 4), (2, 15, 300), (2, 31, 20), (2, 31, 700), (2, 63, 6), (2, 127, 4),
                                    (3, 7, 10), (3, 15, 30), (3, 31, 2)])
def test_sine_transforms(d, m1, n, precision, tol):
    _check(d, m1, n, "fst", precision, tol)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5), ("bf16s", 3e-2)])
@pytest.mark.parametrize("m1,n", [(63, 8), (127, 16), (127, 33)])
def test_corrections(m1, n, precision, tol):
    _check(2, m1, n, "mg", precision, tol)

"""Time transforms of lengths that are not powers of two (the chirp-z method from n = 24,
the direct sum below): preconditioner apply against the oracle.  FP64 1e-12 and FP32 1e-5 as
for the power-of-two transforms (the chirp adds two products and one more transform of
the same kind); BF16 storage 3e-2, the storage's own rounding."""
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


# both sides of the switch (15, 23, 24), every M = 64 .. 8192 with n at both ends of its range,
# one and several columns a CTA, columns left over (m1 = 3, 7, 15: 9, 49, 225 points), 3D
@pytest.mark.parametrize("d,m1,n", [(2, 15, 15), (2, 15, 23), (2, 7, 24), (2, 15, 31), (2, 15, 33), (2, 7, 63),
                                    (2, 31, 65), (2, 15, 100), (2, 7, 127), (2, 7, 129), (2, 7, 255), (2, 7, 257),
                                    (2, 3, 511), (2, 3, 513), (2, 3, 1023), (2, 3, 1025), (2, 3, 2047), (2, 3, 2049),
                                    (2, 1, 4095), (3, 7, 21)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5), ("bf16s", 3e-2)])
@pytest.mark.parametrize("spatial", ["fst", "mg"])
def test_apply_matches_oracle(d, m1, n, spatial, precision, tol):
    if spatial == "fst" and precision == "bf16s":
        pytest.skip("no BF16 storage without multigrid")
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

"""Krylov spaces of every small size and of more steps than the back substitution stages in
shared memory: the iterate after k steps minimises the residual over the k-dimensional
space, so its true residual equals the estimate the Givens rotations give for it (both FP64;
they agree to the orthogonality of the basis, 1e-6 at worst by the re-orthogonalisation
trigger, relative to the initial residual far less)."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_22686_gb300 import build
    build.build()
    assert torch.cuda.is_available()


# 1..17: every count of vectors a projection launch takes, and the second launch; 72 and 73:
# the last staged back substitution and the first that reads H directly; eps = 1 converges
# slowly enough for that many steps
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("k", list(range(1, 18)) + [33, 72, 73, 90])
def test_iterate_has_the_estimated_residual(k, precision):
    from paper_2410_22686_gb300 import Solver
    m1, n = 31, 32
    a = np.exp(0.5 * S.random_vector((m1 + 2, m1 + 2), 2))
    sol = Solver(2, m1, n, 1.0, 1e-4, 1.0, a, spatial="mg", precision=precision, max_iter=96, tiles=None)
    b = torch.from_numpy(S.random_vector((2, n, m1, m1), 3)).cuda()
    x, it, rr = sol.solve(b, rtol=1e-13, maxit=k, raise_on_nonconv=False)
    hist = sol.residual_history()
    r = b - sol.matvec(x)
    true = float(r.norm() / b.norm())
    assert abs(true - rr) <= 1e-12
    if it == k:  # not converged before
        assert len(hist) == k + 1
        assert abs(true - hist[-1]) <= 1e-6 * hist[-1] + 1e-12
    sol.close()

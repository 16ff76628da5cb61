"""The double-float basis where its tiles of 256 unknowns end: last tiles that hold 2 and 254 of
them, and projections over one to four chunks of vectors in less than one tile, in a few and in
many, each run for all its steps (slowly converging problems: eps = 1, a rough coefficient)."""
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


# 2 n m1^2 unknowns, 254 (n m1^2 = 127 mod 128) and 2 modulo 256.  Both bases stop at a true residual of
# 1e-10, and two solutions with that residual differ by at most 2e-10 times the condition of
# A P^{-1} (about 10; 1e-7 is the bound of the mixed path, tests/test_gpu_second_pass.py)
@pytest.mark.parametrize("m1,n", [(3, 71), (31, 63), (63, 127), (1, 127), (31, 65), (63, 129)])
def test_solution_is_the_strict_basis_one(m1, n):
    from paper_2410_22686_gb300 import Solver
    assert 2 * n * m1 * m1 % 256 in (2, 254)
    a = np.exp(0.5 * S.random_vector((m1 + 2, m1 + 2), 2))
    sol = Solver(2, m1, n, 1.0, 1e-2, float(np.sqrt(1 / (n + 1))), a, spatial="mg", precision="fp32", max_iter=80,
                 tiles=None)
    b = torch.from_numpy(S.random_vector((2, n, m1, m1), 3)).cuda()
    x, it, rr = sol.solve(b, rtol=1e-10)
    sol.set_arnoldi("fp64-strict")
    xs, its, rrs = sol.solve(b, rtol=1e-10)
    sol.close()
    assert rr <= 1e-10 and rrs <= 1e-10
    assert abs(it - its) <= 1
    assert float((x - xs).norm() / xs.norm()) <= 1e-7


# The estimate of each step is that of the strict FP64 basis (5%: FP32 roundings of the basis
# vectors differ, a lost or repeated projection shows at once).  The true residual says less
# here: with this coefficient the product's own rounding, u |A| |x|, reaches 1e-6 of it in every
# basis.
@pytest.mark.parametrize("k", [16, 17, 33, 50])
@pytest.mark.parametrize("d,m1,n,gamma", [(2, 7, 2, 1e-2), (2, 15, 1, 1e-2), (3, 7, 8, 1e-4), (2, 31, 64, 1e-4)])
def test_every_step_projects(d, m1, n, gamma, k):
    from paper_2410_22686_gb300 import Solver
    a = np.exp(2.5 * S.random_vector((m1 + 2,) * d, 2))
    sol = Solver(d, m1, n, 1.0, gamma, 1.0, a, spatial="mg", precision="fp32", max_iter=64, tiles=None)
    b = torch.from_numpy(S.random_vector((2, n) + (m1,) * d, 3)).cuda()
    runs = []
    for solve in (sol.solve, sol.solve_graph):
        _, it, _ = solve(b, rtol=1e-13, maxit=k, raise_on_nonconv=False)
        assert it == k
        runs.append(np.array(sol.residual_history()))
    sol.set_arnoldi("fp64-strict")
    _, it, _ = sol.solve(b, rtol=1e-13, maxit=k, raise_on_nonconv=False)
    strict = np.array(sol.residual_history())
    sol.close()
    assert it == k and len(strict) == k + 1
    for hist in runs:
        assert len(hist) == k + 1
        assert (np.abs(hist - strict) <= 0.05 * strict).all()

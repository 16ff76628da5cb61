"""The streamed projections of the double-float basis where their loops end: fewer unknowns than
a tile, a last tile that is not full, less and more than one tile a CTA, and one to four chunks
of vectors in a launch.  As for the other projections, the iterate after k steps has the
residual its Givens rotations give, and the graph-launched solve has the host-driven one's."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [16, 17, 33, 50])
@pytest.mark.parametrize("dim,m1,n", [(2, 3, 2), (2, 7, 4), (2, 15, 16), (3, 7, 16), (2, 31, 64), (2, 63, 32)])
def test_iterate_has_the_estimated_residual(dim, m1, n, k):
    from paper_2410_22686_gb300 import Solver
    a = np.exp(0.5 * S.random_vector((m1 + 2,) * dim, 2))
    sol = Solver(dim, m1, n, 1.0, 1e-4, 1.0, a, spatial="mg", precision="fp32", max_iter=64, tiles=None)
    b = torch.from_numpy(S.random_vector((2, n) + (m1,) * dim, 3)).cuda()
    x, it, rr = sol.solve(b, rtol=1e-13, maxit=k, raise_on_nonconv=False)
    hist = sol.residual_history()
    true = float((b - sol.matvec(x)).norm() / b.norm())
    assert abs(true - rr) <= 1e-12
    if it == k:
        assert abs(true - hist[-1]) <= 1e-6 * hist[-1] + 1e-12
    xg, itg, rg = sol.solve_graph(b, rtol=1e-13, maxit=k, raise_on_nonconv=False)
    trueg = float((b - sol.matvec(xg)).norm() / b.norm())
    assert abs(trueg - rg) <= 1e-12
    if it == k and itg == k:
        assert abs(trueg - true) <= 1e-6 * true + 1e-12
    sol.close()

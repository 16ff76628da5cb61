"""The tuner tries the numbers of time blocks a thread that the built-in rules take: at a small grid,
where eight blocks a thread leave most of the chip idle (31^2 x 64: 32 CTAs, about half as many
as are needed), it finds a shorter one, and the product keeps its values to rounding (the same
terms in the same order, but for the compiler's freedom between kernels: 1e-14)."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_small_grids_take_short_chunks(precision):
    from paper_2410_22686_gb300 import Solver
    m1, n = 31, 64
    a = np.exp(0.3 * S.random_vector((m1 + 2, m1 + 2), 4))
    sol = Solver(2, m1, n, 1.0, 1e-3, 0.3, a, spatial="mg", precision=precision, max_iter=2, tiles=None)
    x = torch.from_numpy(S.random_vector((2, n, m1, m1), 9)).cuda()
    y = sol.matvec(x)
    assert 1 <= sol.autotune(20)["mv_tj"] < 8
    assert float((sol.matvec(x) - y).abs().max()) <= 1e-14 * float(y.abs().max())
    sol.close()

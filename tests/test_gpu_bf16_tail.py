"""BF16 storage with the lower multigrid cycle in one launch: from 63^2 down the iterates stay in
FP32 and are rounded to BF16 once, so the apply differs from the FP32 one by a relative 2^-9 a
value of the planes, at most 1 / eps times that after the time transforms' scaling."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m1,n", [(1, 4), (3, 8), (31, 17), (63, 8)])
def test_one_rounding_from_63_down(m1, n):
    from paper_2410_22686_gb300 import Solver
    a = np.exp(0.5 * S.random_vector((m1 + 2, m1 + 2), 5))
    v = torch.from_numpy(S.random_vector((2, n, m1, m1), 6)).cuda()
    w = {}
    for precision in ("fp32", "bf16s"):
        sol = Solver(2, m1, n, 1.0, 1e-4, 0.25, a, spatial="mg", precision=precision, max_iter=4, tiles=None)
        w[precision] = sol.apply_precond(v)
        sol.close()
    assert float((w["bf16s"] - w["fp32"]).norm()) <= 4 * 2.0 ** -9 * float(w["fp32"].norm())

"""The 3D element multigrid on grids whose rows are too wide for strips in FP64 (511 points): the
per-colour, per-level kernels there against FP32's strips, 1e-5 as between the precisions of the
smaller grids (tests/test_gpu_femg.py)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_levels_too_wide_for_strips_agree_with_strips():
    from paper_2410_22686_gb300 import Solver
    m1 = 511
    x = np.linspace(0.0, 1.0, m1 + 2)
    a = (1.0 + 0.8 * np.sin(9 * x))[:, None, None] * (1.2 + np.cos(7 * x))[:, None] * (1.0 + x)
    a[1::2, ::3, ::2] *= 3.0  # not smooth either
    g = torch.Generator(device="cuda").manual_seed(3)
    v = torch.randn((2, 1, m1, m1, m1), generator=g, dtype=torch.float64, device="cuda")
    w = []
    for precision in ("fp32", "fp64"):
        sol = Solver(3, m1, 1, 1.0, 1e-3, 0.3, a, spatial="mg", precision=precision, max_iter=1, space="fe", tiles=None)
        w.append(sol.apply_precond(v))
        sol.close()
    assert float((w[0] - w[1]).abs().max()) <= 1e-5 * float(w[1].abs().max())

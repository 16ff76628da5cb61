"""Solutions of solves preconditioned in FP32 or with BF16 storage, against stored ones (GB300).
Where the spatial solve is exact, FP32 rounding amplified by A is all that is left of the
residual at rtol, and BF16 storage rounds at 2^-9; so the solution below rtol is what the order
of the preconditioner's FP32 operations makes it.  Any other order is as accurate, but moves
solutions by up to rtol (1e-8) from one version to the next; with these operations kept they
agree to 1e-10 (BF16: 3e-10; the FP64 sums of an iteration may round otherwise).  1e-9 is
between the two."""
import numpy as np
import pytest
import torch

import synthetic as S
from conftest import read_golden

pytestmark = pytest.mark.gpu

# register FFTs along time and space, dense sine products,
# direct sums along time, 3D;
# levels stored in BF16
CASES = [(2, 31, 16, "fp32", 1e-8), (2, 31, 64, "fp32", 1e-8), (2, 31, 128, "fp32", 1e-8), (2, 45, 16, "fp32", 1e-8),
         (2, 30, 8, "fp32", 1e-8), (2, 31, 33, "fp32", 1e-8), (2, 30, 50, "fp32", 1e-8), (3, 15, 33, "fp32", 1e-8),
         (2, 31, 64, "bf16s", 1e-8), (2, 31, 33, "bf16s", 1e-8)]


def solution(d, m1, n, precision, gamma):
    """64 values of the solution for a smooth target."""
    from paper_2410_22686_gb300 import Solver
    x = np.arange(1, m1 + 1) / (m1 + 1)
    t = np.arange(1, n + 1).reshape((n,) + (1,) * d) / (n + 1)
    c = S.random_vector((4,) * (d + 1), 21)
    g = np.zeros((n,) + (m1,) * d)
    for k in np.ndindex(*c.shape):
        f = np.cos(np.pi * k[0] * t)
        for ax in range(d):
            f = f * np.sin(np.pi * (k[1 + ax] + 1) * x).reshape([-1 if q == 1 + ax else 1 for q in range(d + 1)])
        g += c[k] * f
    mg = precision == "bf16s"
    z = np.arange(m1 + 2) / (m1 + 1)
    a = 2.0 ** (np.sin(2 * np.pi * z)[:, None] * np.cos(np.pi * z)[None, :]) if mg else None
    sol = Solver(d, m1, n, 1.0, gamma, float(np.sqrt(1.0 / (n + 1))), a, spatial="mg" if mg else "fst",
                 precision=precision, max_iter=60, tiles=None)
    u = sol.solve(sol.build_rhs(None, torch.from_numpy(g).cuda()), rtol=1e-8)[0].flatten()
    sol.close()
    at = (np.arange(64) * (u.numel() - 1)) // 63
    return u[torch.from_numpy(at).cuda()].cpu().numpy()


@pytest.mark.parametrize("case", range(len(CASES)))
def test_solution_is_the_stored_one(case):
    ref = np.array([float(r[case]) for r in read_golden("fp32_solutions.txt")])
    got = solution(*CASES[case])
    assert np.linalg.norm(got - ref) <= 1e-9 * np.linalg.norm(ref)

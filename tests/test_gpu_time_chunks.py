"""All-at-once products with the built-in number of time blocks per thread: chunk ends,
remainders and chunks of one block, against the oracle (FP64 1e-12: the same formulas in
FP64, summed in another order; FP32 inputs in double-float arithmetic 1e-11: 2^-46 of the
largest term times the few terms of a row)."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import fe as ofe, system as osy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_22686_gb300 import build
    build.build()
    assert torch.cuda.is_available()


def _rel(got, ref):
    return np.abs(got - ref).max() / max(np.abs(ref).max(), 1e-300)


# the differences: a few CTAs a chunk (one block a thread), chunks of 2 and 4 with a
# remainder, n below one chunk; 255^2 x 37 and 31^3 x 37 keep the longest chunks (16)
@pytest.mark.parametrize("d,m1,n", [(2, 7, 5), (2, 31, 3), (2, 63, 1), (2, 127, 17), (2, 255, 37), (3, 15, 7),
                                    (3, 31, 37)])
def test_difference_products(d, m1, n):
    from paper_2410_22686_gb300 import Solver
    a = np.exp(0.3 * S.random_vector((m1 + 2,) * d, 4))
    sol = Solver(d, m1, n, 1.0, 1e-3, 0.3, a, spatial="mg", precision="fp32", max_iter=2, tiles=None)
    x = S.random_vector((2, n) + (m1,) * d, 9)
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, 1e-3)
    dx = torch.from_numpy(x).cuda()
    assert _rel(sol.matvec(dx).cpu().numpy(), osy.apply_A(x, a, tau, alpha)) <= 1e-12
    assert _rel(sol.matvec(dx, transpose=True).cpu().numpy(), osy.apply_AT(x, a, tau, alpha)) <= 1e-12
    x32 = x.astype(np.float32)
    y = sol.matvec_f32(torch.from_numpy(x32).cuda()).cpu().numpy()
    assert _rel(y, osy.apply_A(x32.astype(np.float64), a, tau, alpha)) <= 1e-11
    sol.close()


@pytest.mark.parametrize("d,m1,n", [(2, 13, 5), (2, 61, 3), (2, 250, 37), (3, 6, 9), (3, 30, 33)])
def test_element_products(d, m1, n):
    from paper_2410_22686_gb300 import Solver
    sol = Solver(d, m1, n, 1.0, 1e-3, 0.3, None, spatial="fst", precision="fp32", max_iter=2, space="fe", tiles=None)
    M, K = ofe.fe_matrices(m1, d)
    x = S.random_vector((2, n) + (m1,) * d, 9)
    tau, alpha = osy.time_step(1.0, n), osy.alpha_weight(1.0, n, 1e-3)
    dx = torch.from_numpy(x).cuda()
    assert _rel(sol.matvec(dx).cpu().numpy(), ofe.apply_A(x, M, K, tau, alpha)) <= 1e-12
    assert _rel(sol.matvec(dx, transpose=True).cpu().numpy(), ofe.apply_AT(x, M, K, tau, alpha)) <= 1e-12
    x32 = x.astype(np.float32)
    y = sol.matvec_f32(torch.from_numpy(x32).cuda()).cpu().numpy()
    assert _rel(y, ofe.apply_A(x32.astype(np.float64), M, K, tau, alpha)) <= 1e-11
    sol.close()

"""The element product of an FP32 vector with a nodal coefficient (double-float sums, widened on
the integer pipes) against the FP64 product of the same values, over chunk lengths of time that
do and do not divide n, one block per chunk, and scales of tau, alpha and x that move the
product's terms against each other by many orders of magnitude."""
import pytest
import torch

from paper_2410_22686_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,m1,n", [(2, 3, 2), (2, 31, 17), (2, 63, 64), (2, 127, 37), (2, 255, 5), (3, 3, 2),
                                      (3, 7, 33), (3, 15, 13), (3, 31, 64)])
@pytest.mark.parametrize("T,gamma,scale", [(1.0, 1e-4, 1.0), (100.0, 1e-8, 1e-12), (1e-3, 1.0, 1e12)])
def test_fp32_product_matches_fp64(dim, m1, n, T, gamma, scale):
    gen = torch.Generator().manual_seed(m1 * 100 + n)
    a = torch.exp(0.5 * torch.randn((m1 + 2,) * dim, generator=gen, dtype=torch.float64)).numpy()
    sol = Solver(dim, m1, n, T, gamma, 0.1, a, precision="fp32", max_iter=4, space="fe")
    x = (scale * torch.randn((2, n) + (m1,) * dim, generator=gen)).to(torch.float32).cuda()
    y = sol.matvec_f32(x)
    ref = sol.matvec(x.double())
    # random x: an output's terms sum to less than 64 times the largest output in magnitude
    # (27 terms of at most the centre's); 2^-44 of them, plus the FP64 product's own 2^-50
    assert torch.isfinite(y).all()
    assert float((y - ref).abs().max()) <= 64 * 2.0 ** -44 * float(ref.abs().max())
    zero = sol.matvec_f32(torch.zeros_like(x))
    assert not zero.any()

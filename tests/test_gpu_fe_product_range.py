"""The element product of an FP32 vector with a nodal coefficient at the ends of its range: K entries
up to the largest FP32 value (they are kept in FP32 pairs, scaled by no more than one) and steps
of time beyond the exponents the pairs' conversion holds (FP64 arithmetic there), against the FP64
product: 64 2^-44 of the largest output, as tests/test_gpu_fe_product.py derives it."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# 8/3 a (2D) and 32 a (3D) are the largest K entries: 2.7e38 of 3.4e38; tau = T / (n + 1) with a
# fraction above one half
@pytest.mark.parametrize("dim,m1,n,T,level,scale", [(2, 15, 17, 1.0, 1e38, 1e-4), (3, 7, 8, 1.0, 8.5e36, 1e-4),
                                                    (2, 15, 17, 1e-290, 1.0, 1.0), (3, 7, 8, 1e-290, 1.0, 1.0),
                                                    (2, 15, 17, 1e-272, 1.0, 1e-30), (2, 15, 17, 1e290, 1.0, 1.0),
                                                    (3, 7, 8, 1e290, 1.0, 1.0)])
def test_fp32_product_matches_fp64(dim, m1, n, T, level, scale):
    from paper_2410_22686_gb300 import Solver
    gen = torch.Generator().manual_seed(7)
    a = level * torch.exp(-0.5 * torch.rand((m1 + 2,) * dim, generator=gen, dtype=torch.float64)).numpy()
    sol = Solver(dim, m1, n, T, 1.0, 0.1, a, precision="fp32", max_iter=4, space="fe", tiles=None)
    x = (scale * torch.randn((2, n) + (m1,) * dim, generator=gen)).to(torch.float32).cuda()
    y, ref = sol.matvec_f32(x), sol.matvec(x.double())
    sol.close()
    assert torch.isfinite(ref).all()
    assert float((y - ref).abs().max()) <= 64 * 2.0 ** -44 * float(ref.abs().max())

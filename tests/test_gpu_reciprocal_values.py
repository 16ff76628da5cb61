"""The FP64 reciprocal of the shifted diagonals, value by value: inside the FP32 normal range an FP32
seed with an error e <= 2^-21 and one cubic step, whose remainder e^3 is far below the last
place, so the last rounding alone is left: within one unit in the last place of 1 / d (the
correctly rounded quotient).  A step without the cubic term would be 2^10 units off.
Outside that range, signs and the values without a reciprocal take the division itself."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _reciprocal(d):
    from paper_2410_22686_gb300 import capi
    t = torch.from_numpy(np.ascontiguousarray(d)).cuda()
    r = torch.empty_like(t)
    capi.check(capi.load().pc_selftest_reciprocal(ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(r.data_ptr()), t.numel(),
                                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return r.cpu().numpy()


# both ends of the fast range [2^-124, 2^124) and what lies beyond them, the middle
@pytest.mark.parametrize("exponents", [(-127, -121), (-3, 3), (120, 127), (-1000, 1000)])
def test_within_one_unit_of_the_quotient(exponents):
    rng = np.random.default_rng(5)
    m = np.concatenate([1.0 + rng.random(200000), [1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52, 1.5]])
    for e in range(exponents[0], exponents[1] + 1, max(1, (exponents[1] - exponents[0]) // 6)):
        d = np.ldexp(m, e)
        ref = 1.0 / d
        assert (np.abs(_reciprocal(d) - ref) <= np.spacing(ref)).all(), e


def test_other_values_divide():
    d = np.array([0.0, -0.0, -1.0, -3.0, np.inf, -np.inf, 2.0 ** -1074, 1e-310, 1.7e308])
    with np.errstate(divide="ignore", over="ignore"):
        ref = 1.0 / d
    assert (_reciprocal(d) == ref).all()
    assert np.isnan(_reciprocal(np.array([np.nan]))).all()

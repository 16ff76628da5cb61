"""The FP64 difference product of vectors smooth in time where tau K is small against the identity:
the difference of neighbouring time blocks is formed before tau K v is added, so an output's
error is that of its terms and not that of the block itself.  Elementwise, with u = 2^-53 and
E = d |v| + sum of w |neighbours|: the 2 dim + 1 terms of tau K v and their sum (2 dim + 2
roundings), the coefficients (4: mean, division by h^2, product with tau, diagonal's sum), the
time difference, its sum with tau K v and the one with alpha x (3): u (16 E + 3 |difference| +
2 alpha |x|).  The reference is in extended precision."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _terms(v, a, tau, h):
    """tau K v and E, extended precision."""
    d = v.ndim - 1
    inner = (slice(1, -1),) * d
    out, size = np.zeros_like(v), np.zeros_like(v)
    p = np.pad(v, [(0, 0)] + [(1, 1)] * d)
    for b in range(d):
        for step in (slice(0, -2), slice(2, None)):
            e = inner[:b] + (step,) + inner[b + 1:]
            w = tau * (a[inner] + a[e]) / 2 / h ** 2
            out += w * (v - p[(slice(None),) + e])
            size += w * (np.abs(v) + np.abs(p[(slice(None),) + e]))
    return out, size


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("d,m1,n,T", [(2, 15, 255, 3e-3), (2, 7, 1023, 1e-2), (3, 7, 255, 3e-3)])
def test_error_is_that_of_the_terms(d, m1, n, T, transpose):
    from paper_2410_22686_gb300 import Solver
    L = np.longdouble
    a = np.exp(0.3 * S.random_vector((m1 + 2,) * d, 4))
    t = (np.arange(1, n + 1) / (n + 1)).reshape((n,) + (1,) * d)
    x = np.stack([np.cos(t + S.random_vector((1,) + (m1,) * d, k)) for k in (5, 6)])
    sol = Solver(d, m1, n, T, 1.0, 0.3, a, spatial="mg", max_iter=2, tiles=None)
    y = sol.matvec(torch.from_numpy(x).cuda(), transpose=transpose).cpu().numpy()
    sol.close()
    x, a = x.astype(L), a.astype(L)
    tau, h = L(T) / (n + 1), L(1) / (m1 + 1)
    alpha = tau  # gamma = 1
    k, size = zip(*(_terms(v, a, tau, h) for v in x))
    zero = np.zeros_like(x[0][:1])
    diff = [x[1] - np.concatenate([x[1][1:], zero]), x[0] - np.concatenate([zero, x[0][:-1]])]
    sg = -1 if transpose else 1
    ref = np.stack([alpha * x[0] + sg * (diff[0] + k[1]), alpha * x[1] - sg * (diff[1] + k[0])])
    bound = 2.0 ** -53 * np.stack([16 * size[1 - i] + 3 * np.abs(diff[i]) + 2 * alpha * np.abs(x[i]) for i in (0, 1)])
    assert (np.abs(y - ref) <= bound).all()

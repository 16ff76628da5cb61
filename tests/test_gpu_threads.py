"""Two threads with a handle each, of different shapes, so that the same kernels are launched with
different amounts of shared memory at the same time: every call succeeds and gives the values
the handle gives alone."""
import threading

import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


# chirp-z; direct sums; sine products; element multigrid in 2D (strips, small levels) and 3D;
# the lower cycle from 31^2 and in place from 63^2
@pytest.mark.parametrize("one,two,more", [
    ((2, 7, 100), (2, 7, 2049), dict(spatial="fst")),
    ((2, 12, 50), (2, 12, 700), dict(spatial="fst", precision="fp32")),
    ((2, 20, 4), (2, 300, 4), dict(spatial="fst")),
    ((2, 63, 4), (2, 127, 4), dict(spatial="mg", space="fe")),
    ((2, 15, 8), (2, 63, 8), dict(spatial="mg", space="fe", precision="fp32")),
    ((3, 7, 4), (3, 31, 4), dict(spatial="mg", space="fe")),
    ((2, 7, 8), (2, 31, 8), dict(spatial="mg")),
    ((2, 15, 8), (2, 63, 8), dict(spatial="mg", precision="fp32")),
])
def test_applies_of_two_handles_at_once(one, two, more):
    from paper_2410_22686_gb300 import Solver
    sols, vs, refs = [], [], []
    for k, (d, m1, n) in enumerate((one, two)):
        a = None if more["spatial"] == "fst" else np.exp(0.3 * S.random_vector((m1 + 2,) * d, k))
        sols.append(Solver(d, m1, n, 1.0, 1e-4, 0.25, a, max_iter=2, tiles=None, **more))
        vs.append(torch.from_numpy(S.random_vector((2, n) + (m1,) * d, 7 + k)).cuda())
        refs.append(sols[k].apply_precond(vs[k]))
    torch.cuda.synchronize()
    outs, errors, start = [torch.empty_like(v) for v in vs], [], threading.Barrier(2)

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(400):
                    sols[k].apply_precond(vs[k], out=outs[k])
                torch.cuda.current_stream().synchronize()
        except Exception as ex:  # noqa: BLE001 - reported by the main thread
            errors.append(repr(ex))

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in sols:
        s.close()
    assert not errors
    for k in (0, 1):
        assert torch.equal(outs[k], refs[k])

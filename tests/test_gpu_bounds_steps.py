"""A bounds call of few Lanczos steps costs the same whatever the context ran
before: the tridiagonal extremes take shared memory for the steps of the call,
not for the most steps the context has seen (512 of them leave one warp per SM).
Small regions, so that the extremes are a good part of the call; 10 % is far above
the spread of the fastest of ten."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_short_call_after_a_long_one():
    import torch
    from paper_1708_07913_gb300 import SQ_FP32, SQSolver
    shape = (48, 49, 50)
    V = torch.from_numpy(-1.0 - 0.8 * np.random.default_rng(3).random(int(np.prod(shape)))).cuda()
    s = SQSolver(shape, 0.5, 1.01, 8, SQ_FP32)

    def best():
        t = 1e30
        for _ in range(10):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            s.bounds(V, 40, 0.01)
            e1.record()
            torch.cuda.synchronize()
            t = min(t, e0.elapsed_time(e1))
        return t, s.chi.clone(), s.zeta.clone()

    best()
    t0, c0, z0 = best()
    s.bounds(V, 512, 0.01)
    t1, c1, z1 = best()
    s.close()
    assert torch.equal(c0, c1) and torch.equal(z0, z1)
    assert t1 <= 1.1 * t0, (t0, t1)

"""The SM-share plan of a batch of one system gives it the whole GPU, so it is
no slower than the plain stream plan: both region kernels take their own
resident CTAs (with projectors below 23^3 moments run one CTA per SM, Lanczos
several).  Cut to the moments' count, Lanczos would take more than twice as long;
20 % is far above the spread of a step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _step_ms(batch, args):
    import torch
    best = 1e30
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        batch.run(*args, n_lanczos=40, margin=0.02)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    batch.results()
    return best


@pytest.mark.parametrize("m", [7, 9])
def test_share_of_one_system_is_the_whole_gpu(monkeypatch, m):
    import torch
    from paper_1708_07913_gb300 import SQ_FP32, SQBatch, SQSolver, sq
    from test_gpu_quad import _inputs
    monkeypatch.delenv("SQ_REGION_KERNEL", raising=False)
    shape, h = (17, 16, 15), 0.5
    pos, V, proj = _inputs(shape, h, 3, 30 + m)
    s = SQSolver(shape, h, (m + 0.25) * h, 16, SQ_FP32, pos, proj)
    args = ([torch.from_numpy(V).cuda()], [float(np.prod(shape)) * 0.1], [0.2])
    ms = {}
    for plan in (sq.SQ_BATCH_STREAMS, sq.SQ_BATCH_STREAMS_SHARE):
        b = SQBatch([s])
        b.set_plan(plan)
        ms[plan] = _step_ms(b, args)
        b.close()
    s.close()
    assert ms[sq.SQ_BATCH_STREAMS_SHARE] <= 1.2 * ms[sq.SQ_BATCH_STREAMS], ms

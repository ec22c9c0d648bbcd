"""A batch run after its contexts' buffers moved: a bounds call of more Lanczos
steps replaces the coefficient buffers, and the queue plan of another batch can
replace the per-CTA scratch.  The batch's next run uses the new ones and gives the
same results bit for bit (local systems, fixed order everywhere)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["SQ_FP32", "SQ_FP64"])
@pytest.mark.parametrize("plan", ["SQ_BATCH_STREAMS", "SQ_BATCH_QUEUE"])
def test_run_after_buffers_moved(plan, prec):
    import torch
    import paper_1708_07913_gb300 as P
    from paper_1708_07913_gb300 import SQBatch, SQSolver, sq
    rng = np.random.default_rng(4)
    solvers, Vs, ne = [], [], []
    for shape, m in (((6, 5, 7), 3), ((9, 8, 10), 5)):
        solvers.append(SQSolver(shape, 0.5, (m + 0.25) * 0.5, 16, getattr(P, prec)))
        Vs.append(torch.from_numpy(-1.0 - 0.8 * rng.random(int(np.prod(shape)))).cuda())
        ne.append(0.2 * Vs[-1].numel())
    b = SQBatch(solvers)
    b.set_plan(getattr(sq, plan), 1)

    def run():
        for s in solvers:
            s.rho.zero_()
        b.run(Vs, ne, [0.2, 0.2], n_lanczos=12, margin=0.05)
        b.results()
        return [t.clone() for s in solvers for t in (s.chi, s.zeta, s.moments, s.rho)]

    first = run()
    for s, V in zip(solvers, Vs):
        s.bounds(V, 40, 0.05)
    other = SQBatch(solvers)
    other.set_plan(sq.SQ_BATCH_QUEUE, 4)
    other.run(Vs, ne, [0.2, 0.2], n_lanczos=40, margin=0.05)
    other.results()
    for x, y in zip(first, run()):
        assert torch.equal(x, y)
    b.close()
    other.close()
    for s in solvers:
        s.close()

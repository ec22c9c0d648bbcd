"""The Fermi search runs until its bracket closes in FP64, however small the
level is against the spectrum: one middle zero x of T_5 (6e-17) holds half of the
electrons, the temperature is so low that the count is a step, and the level has
to land on chi + zeta x itself.  A bracket of the width of the spectrum halved 56
times is still 1e-17 wide.  Tolerances: the spacing of FP64 numbers at the level
(4e-28 at 3e-12) and 41 kT; 1e-24 where the level comes from Lanczos bounds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

X2 = float(np.cos(np.pi * 2.5 / 5))
SHAPES = [(3, 5, 2), (40, 42, 41)]                       # three points per pass, and one


@pytest.mark.parametrize("shape", SHAPES)
def test_single_system(shape):
    import torch
    from paper_1708_07913_gb300 import SQ_FP64, SQSolver, sq
    nq = int(np.prod(shape))
    s = SQSolver(shape, 0.5, 0.5, 4, SQ_FP64)
    chi = torch.full((nq,), 3e-12, dtype=torch.float64, device="cuda")
    zeta = torch.ones_like(chi)
    mom = torch.zeros(nq, 5, dtype=torch.float64, device="cuda")
    mom[:, 0] = 1.0                                      # equal weights at the five zeros
    mu = sq.sq_fermi_level(s.ctx, mom, chi, zeta, float(nq), 1e-30)
    s.close()
    assert abs(mu - (3e-12 + X2)) <= 1e-26


@pytest.mark.parametrize("plan", ["SQ_BATCH_STREAMS", "SQ_BATCH_QUEUE"])
@pytest.mark.parametrize("shape", SHAPES)
def test_captured_batch(shape, plan):
    """Regions of one point: chi is the level itself, zeta the margin, and every
    moment that of the middle zero."""
    import torch
    from paper_1708_07913_gb300 import SQ_FP64, SQBatch, SQSolver, sq
    nq, h = int(np.prod(shape)), 0.5
    s = SQSolver(shape, h, 0.1 * h, 4, SQ_FP64)
    w0 = -sum(1.0 / q ** 2 for q in range(1, 7)) / h ** 2
    V = torch.full((nq,), 3.0 * w0 + 1e-13, dtype=torch.float64, device="cuda")
    b = SQBatch([s])
    b.set_plan(getattr(sq, plan), 1)
    b.run([V], [float(nq)], [1e-30], n_lanczos=4, margin=0.5)
    mu = b.results()[0]["mu"]
    chi, zeta = s.chi.cpu().numpy(), s.zeta.cpu().numpy()
    b.close()
    s.close()
    assert np.all(chi == chi[0]) and abs(chi[0]) < 1e-12
    assert abs(mu - (chi[0] + zeta[0] * X2)) <= 1e-24

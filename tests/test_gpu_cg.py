"""Conjugate gradients of sq_poisson and sq_kerker on the edges of their
range: axes shorter than the half order of the differences (6: a neighbour
wraps more than once), of exactly that and of one more, and an iteration count
beyond one lot of launches.  Reference: the spectral solution.

Tolerance.  The residual is below 1e-13 |f|; the error of the solution exceeds
it by at most the condition number of the operator on the mean-free grid
functions, which is taken from the symbol, times a few roundings."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1708_07913_gb300 import SQ_FP64, SQSolver, build, sq  # noqa: E402

build()
DEV = "cuda:0"


def _axis(n, h):
    w = oracle.fd_weights(6, h)
    th = 2 * np.pi * np.fft.fftfreq(n)
    return -(2 * w[0] + 2 * sum(w[d] * np.cos(d * th) for d in range(1, 7)))


@pytest.mark.parametrize("shape", [(4, 5, 9), (6, 7, 11), (33, 2, 8), (1, 12, 6), (48, 47, 6)])
def test_short_axes_match_the_spectral_solution(shape):
    h = 0.5
    n1, n2, n3 = shape
    solver = SQSolver(shape, h, h + 1e-9, 8, SQ_FP64, np.zeros((0, 3)), (), device=DEV)
    sq.sq_set_stream(solver.ctx)
    S = _axis(n3, h)[:, None, None] + _axis(n2, h)[None, :, None] + _axis(n1, h)[None, None, :]
    rng = np.random.default_rng(sum(shape))
    rho = rng.uniform(0.0, 0.05, size=(n3, n2, n1)) + 0.02 * np.cos(2 * np.pi * np.arange(n1) / n1)[None, None, :]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).to(DEV)
    out = torch.empty(n1 * n2 * n3, dtype=torch.float64, device=DEV)
    S0 = S.copy()
    S0[0, 0, 0] = 1.0
    P = 4 * np.pi * np.fft.fftn(rho - rho.mean()) / S0
    P[0, 0, 0] = 0.0
    ref = np.real(np.fft.ifftn(P))
    cond = S.max() / S.ravel()[1:].min()
    it, res = sq.sq_poisson(solver.ctx, dev(rho), out, 1e-13)
    assert it > 0 and res <= 1e-13
    assert np.linalg.norm(out.cpu().numpy() - ref.ravel()) <= 2e-13 * cond * np.linalg.norm(ref)
    v_in = rng.standard_normal((n3, n2, n1))
    f = 0.1 * rng.standard_normal((n3, n2, n1)) + 0.05
    k0, a = 0.8, 0.2
    sq.sq_kerker(solver.ctx, dev(v_in), dev(v_in + f), k0, a, out, tol=1e-13)
    y = np.real(np.fft.ifftn(np.fft.fftn(f) * (S + a * k0 ** 2) / (S + k0 ** 2)))
    cond = (S.max() + k0 ** 2) / k0 ** 2
    assert np.linalg.norm(out.cpu().numpy() - (v_in + y).ravel()) <= 2e-13 * cond * np.linalg.norm(v_in)
    solver.close()

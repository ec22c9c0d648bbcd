"""Density and energies for intervals of any sign of zeta: [chi - zeta, chi +
zeta] run through backwards (zeta < 0) or a single point (zeta = 0).  The sums run
over the zeros E_k = chi + zeta x_k in every case, as the oracle's do.  Tolerances as in
test_gpu_fermi.py, and the rounding of E_k (1e-14 at most here) over kT."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kT", [2e-3, 0.05, 5.0])
@pytest.mark.parametrize("npl", [4, 24, 48])
def test_density_matches_oracle_for_any_zeta(npl, kT):
    import torch
    from paper_1708_07913_gb300 import SQ_FP64, SQSolver, sq
    shape, h = (7, 6, 5), 0.5
    nq, K = int(np.prod(shape)), npl + 1
    rng = np.random.default_rng(npl)
    W0 = rng.random((nq, K))
    W0 /= W0.sum(1, keepdims=True)
    th = np.pi * (np.arange(K) + 0.5) / K
    mom = W0 @ np.cos(np.outer(th, np.arange(K)))
    chi = 6.0 + rng.random(nq)
    zeta = (20.0 + rng.random(nq)) * rng.choice([-1.0, 1.0], nq)
    zeta[::11] = 0.0
    s = SQSolver(shape, h, h + 1e-9, npl, SQ_FP64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()
    rho = torch.empty(nq, dtype=torch.float64, device="cuda")
    W = oracle.cc_weights(mom)
    tol = 1e-12 + 1e-14 / kT
    for mu in (-3.0, 6.5, 11.0):
        eb, es, n = sq.sq_density_energy(s.ctx, dev(mom).view(nq, K), dev(chi), dev(zeta), mu, kT, rho)
        rho_o, eb_o, es_o, n_o = oracle.density_energy(W, chi, zeta, mu, kT, h)
        np.testing.assert_allclose(rho.cpu().numpy(), rho_o, rtol=0, atol=tol * 2 / h ** 3)
        assert abs(eb - eb_o) <= tol * 2 * nq * 30.0
        assert abs(es - es_o) <= tol * 2 * nq * kT
        assert abs(n - n_o) <= tol * 2 * nq
    s.close()

"""Fermi level, density and energies over the forms of their kernels: one
node, few nodes, and more than 65536 (one search point per pass instead of
three); the smallest and largest n_pl; temperatures far below the spacing of the
Chebyshev zeros and far above it.  The moments are those of positive random
weights, so the electron count is monotone.

Tolerances.  A count is a sum of at most Nd (n_pl + 1) positive terms by trees in
FP64, and the weights are sums of n_pl + 1 cosines: 1e-13 of the electrons, with
the derivative of the count the Fermi level; densities and energies 1e-12 of the
sums of the absolute terms."""
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


@pytest.mark.parametrize("kT", [2e-3, 0.05, 5.0])
@pytest.mark.parametrize("shape,npl", [((1, 1, 1), 4), ((3, 5, 2), 24), ((9, 8, 7), 512), ((16, 16, 16), 48),
                                       ((40, 42, 41), 8)])
def test_search_and_density_match_oracle(shape, npl, kT):
    h = 0.5
    nq, K = int(np.prod(shape)), npl + 1
    rng = np.random.default_rng(nq + npl)
    W0 = rng.random((nq, K))
    W0 /= W0.sum(1, keepdims=True)
    th = np.pi * (np.arange(K) + 0.5) / K
    mom = W0 @ np.cos(np.outer(th, np.arange(K)))
    chi = 6.0 + rng.random(nq)
    zeta = 20.0 + rng.random(nq)
    ne = 0.37 * 2 * nq
    W = oracle.cc_weights(mom)
    mu_o, _ = oracle.fermi_level(W, chi, zeta, ne, kT)
    solver = SQSolver(shape, h, h + 1e-9, npl, SQ_FP64, np.zeros((0, 3)), (), device=DEV)
    sq.sq_set_stream(solver.ctx)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).to(DEV)
    m, c, z = dev(mom).view(nq, K), dev(chi), dev(zeta)
    mu = sq.sq_fermi_level(solver.ctx, m, c, z, ne, kT)
    d = max(1e-10, 1e-3 * kT)
    slope = (oracle.electron_count(W, chi, zeta, mu_o + d, kT) - oracle.electron_count(W, chi, zeta, mu_o - d, kT)) / (2 * d)
    n_at = oracle.electron_count(W, chi, zeta, mu, kT)
    assert abs(n_at - ne) <= 1e-12 * nq + 4 * slope * 4e-15 * 30.0      # in a gap of the count mu itself is free
    rho = torch.empty(nq, dtype=torch.float64, device=DEV)
    eb, es, n = sq.sq_density_energy(solver.ctx, m, c, z, mu, kT, rho)
    rho_o, eb_o, es_o, n_o = oracle.density_energy(W, chi, zeta, mu, kT, h)
    np.testing.assert_allclose(rho.cpu().numpy(), rho_o, rtol=0, atol=1e-12 * 2 / h ** 3)
    assert abs(eb - eb_o) <= 1e-12 * 2 * nq * 30.0
    assert abs(es - es_o) <= 1e-12 * 2 * nq * kT
    assert abs(n - n_o) <= 1e-12 * 2 * nq
    solver.close()

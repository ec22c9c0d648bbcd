"""The FP32 quad kernels against the general single-CTA kernels.

Every region half-width that has a quad kernel, with and without projectors, on
odd and uneven grids (regions larger than the cell among them): the two forms
compute the same sums in FP32 in different orders, so each is within the FP32
form's tolerances of the exact result (2e-5 for moments, 2e-4 relative for the
Lanczos bounds; tests/test_gpu_parity.py) and they are held to the same ones
against each other.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

GRIDS = [(9, 12, 7), (13, 8, 10)]


def _solver(monkeypatch, kernel, shape, h, m, npl, pos, proj):
    from paper_1708_07913_gb300 import SQ_FP32, SQSolver
    if kernel:
        monkeypatch.setenv("SQ_REGION_KERNEL", kernel)
    else:
        monkeypatch.delenv("SQ_REGION_KERNEL", raising=False)
    return SQSolver(shape, h, (m + 0.25) * h, npl, SQ_FP32, pos, proj)


def _inputs(shape, h, atoms, seed, r_nl=3.0):
    rng = np.random.default_rng(seed)
    L = np.array(shape) * h
    pos = rng.uniform(0.0, 1.0, (atoms, 3)) * L
    V = -1.0 - 0.8 * rng.random(shape[0] * shape[1] * shape[2])
    return pos, V, [(0, synth.GAMMA_S, 1.1, r_nl), (1, synth.GAMMA_P, 1.1, r_nl)]


@pytest.mark.parametrize("nonlocal_", [False, True])
@pytest.mark.parametrize("m", range(7, 16))
def test_quad_matches_general(monkeypatch, m, nonlocal_):
    import torch
    shape, h, npl = GRIDS[m % 2], 0.5, 16
    atoms = 1 if m >= 14 else 3                          # few enough for the tables of the candidates to fit
    pos, V, proj = _inputs(shape, h, atoms, 40 + m)
    V = torch.from_numpy(V).cuda()
    out = {}
    for kernel in ("cta", ""):
        s = _solver(monkeypatch, kernel, shape, h, m, npl, pos, proj if nonlocal_ else ())
        chi, zeta = s.bounds(V, 24, 0.02)
        chi, zeta = chi.clone(), zeta.clone()
        if not out:
            bounds = (chi, zeta)
        mom = s.compute_moments(V, *bounds).clone()
        again = s.compute_moments(V, *bounds)
        if not kernel:
            assert torch.equal(mom, again)               # fixed order everywhere
        torch.cuda.synchronize()
        out[kernel] = (chi, zeta, mom)
        s.close()
    (ca, za, ma), (cb, zb, mb) = out["cta"], out[""]
    assert float((ma - mb).abs().max()) < 2e-5
    width = float(za.abs().max())
    assert float((ca - cb).abs().max()) < 2e-4 * width
    assert float((za - zb).abs().max()) < 2e-4 * width


@pytest.mark.parametrize("kernel", ["cta", ""])
def test_too_many_row_entries_refused(monkeypatch, kernel):
    """More than 24 projector entries on a region row are refused by both forms."""
    import torch
    from paper_1708_07913_gb300 import SQError, sq
    shape, h = (10, 9, 11), 0.5
    pos, V, proj = _inputs(shape, h, 11, 5)
    s = _solver(monkeypatch, kernel, shape, h, 7, 8, pos, proj)
    chi = torch.full((s.n_nodes,), 20.0, dtype=torch.float64, device="cuda")
    zeta = torch.full_like(chi, 60.0)
    s.compute_moments(torch.from_numpy(V).cuda(), chi, zeta)
    with pytest.raises(SQError) as e:
        sq.sq_sync(s.ctx)
    assert e.value.code == sq.SQ_ECAPACITY
    s.close()

"""Device memory of a context: the quad kernels' per-CTA scratch in place of the
general kernels', not on top of it, and the general kernels when it cannot be had."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_quad import GRIDS, _inputs  # noqa: E402

MB = 1 << 20


def _setup(monkeypatch, kernel, m, atoms, npl=16):
    """(context, bytes it took)"""
    import torch
    from paper_1708_07913_gb300 import SQ_FP32, sq
    if kernel:
        monkeypatch.setenv("SQ_REGION_KERNEL", kernel)
    else:
        monkeypatch.delenv("SQ_REGION_KERNEL", raising=False)
    shape, h = GRIDS[m % 2], 0.5
    pos, _, proj = _inputs(shape, h, max(atoms, 1), 40 + m)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx = sq.sq_setup_grid(*shape, h, 6, (m + 0.25) * h, npl, SQ_FP32, pos if atoms else None, proj if atoms else ())
    return ctx, free - torch.cuda.mem_get_info()[0]


def _quad_scratch(m, ccap, lb):
    """Per CTA: the potential window, then (with projectors) the lists of a
    (quad, row pair, plane pair), the entries by candidate and, at 31^3, the
    tables that do not fit shared memory."""
    up = lambda b: (b + 255) // 256 * 256
    total = up(4 * (2 * m + 1) * 2 * 32 * 16)
    if ccap:
        total += up(4 * (m + 1) * 96 * 32 * 8) + up(ccap * ((lb * lb + 63) // 64 * 64) * 16)
        if m == 15:
            total += up(ccap * (lb // 2 + 1) * 16) + up((ccap * (lb + 1) + 1) * 16)
    return total


@pytest.mark.parametrize("m,atoms", [(8, 0), (15, 0), (11, 3), (14, 1), (15, 1)])
def test_quad_context_holds_its_own_scratch_only(monkeypatch, m, atoms):
    import torch
    from paper_1708_07913_gb300 import sq
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for _ in range(2):                                   # the first one also loads the kernels
        ctx, took = _setup(monkeypatch, "", m, atoms)
        info = sq.sq_context_info(ctx)
        sq.sq_destroy(ctx)
    assert info["moments"] == info["lanczos"] == sq.FORM_QUAD
    need = _quad_scratch(m, info["ccap"] if atoms else 0, 13)
    assert took <= need * sms + 16 * MB, (took / MB, need * sms / MB)


def test_region_force_form_gets_its_scratch_on_first_use(monkeypatch):
    """A context that runs the quad kernels, asked for the region force form and
    for the quad form again (FP32 tolerance of test_gpu_force.py, twice)."""
    import torch
    from paper_1708_07913_gb300 import sq
    from test_gpu_force import FP32_FORCE
    m = 12
    _, V, _ = _inputs(GRIDS[0], 0.5, 3, 40 + m)
    V = torch.from_numpy(V).cuda()
    ctx, _ = _setup(monkeypatch, "", m, 3)
    chi, zeta = torch.empty_like(V), torch.empty_like(V)
    sq.sq_spectral_bounds(ctx, V, chi, zeta, 24, 0.02)
    F = {}
    for form in ("", "region", ""):
        monkeypatch.setenv("SQ_FORCE_KERNEL", form) if form else monkeypatch.delenv("SQ_FORCE_KERNEL", raising=False)
        F[form] = torch.empty(9, dtype=torch.float64, device="cuda")
        sq.sq_nl_forces(ctx, V, chi, zeta, float(chi.median()), 0.1, F[form])
    sq.sq_destroy(ctx)
    scale = float(F["region"].abs().max())
    assert scale > 1e-6 and float((F[""] - F["region"]).abs().max()) <= 2 * FP32_FORCE * scale


def test_general_kernels_when_the_quad_scratch_cannot_be_had(monkeypatch):
    import torch
    from paper_1708_07913_gb300 import sq
    m, atoms = 14, 1
    shape, h = GRIDS[m % 2], 0.5
    _, V, _ = _inputs(shape, h, 1, 40 + m)
    nq = V.size
    V = torch.from_numpy(V).cuda()
    chi = torch.full((nq,), 20.0, dtype=torch.float64, device="cuda")
    zeta = torch.full_like(chi, 60.0)
    bounds = [torch.empty_like(chi), torch.empty_like(chi)]
    mom = {}
    took = {}
    for kernel in ("", "cta", "", "cta"):                # the first ones also load the kernels
        ctx, took[kernel] = _setup(monkeypatch, kernel, m, atoms)
        mom[kernel] = torch.empty(nq, 17, dtype=torch.float64, device="cuda")
        sq.sq_spectral_bounds(ctx, V, *bounds, 8, 0.02)
        sq.sq_moments(ctx, V, chi, zeta, mom[kernel])
        sq.sq_sync(ctx)
        sq.sq_destroy(ctx)
    assert took[""] > took["cta"] + 80 * MB
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - took["cta"] - 40 * MB, dtype=torch.uint8, device="cuda")
    try:
        ctx, _ = _setup(monkeypatch, "", m, atoms)
        info = sq.sq_context_info(ctx)
        assert info["moments"] == info["lanczos"] == sq.FORM_GENERAL
        sq.sq_moments(ctx, V, chi, zeta, mom[""])
        sq.sq_sync(ctx)
        sq.sq_destroy(ctx)
    finally:
        del ballast
        torch.cuda.empty_cache()
    assert float((mom[""] - mom["cta"]).abs().max()) < 2e-5       # FP32, as in test_gpu_parity.py
    assert np.isfinite(mom[""].cpu().numpy()).all()

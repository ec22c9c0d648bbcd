"""The FP32 quad force kernels against the general region kernel's form.

Every region half-width that has a quad kernel, on odd and uneven grids
(regions larger than the cell, atoms with several images in a region), for all
nodes and for a list of them with repeats: both forms are within the FP32
tolerance of the exact forces (tests/test_gpu_force.py: 1e-4 of the largest
force), so within twice that of each other; the quad form repeats bit for bit."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_force import FP32_FORCE  # noqa: E402
from test_gpu_quad import GRIDS, _inputs, _solver  # noqa: E402


@pytest.mark.parametrize("m", range(7, 16))
def test_quad_forces_match_region_form(monkeypatch, m):
    import torch
    shape, h, npl = GRIDS[m % 2], 0.5, 16
    pos, V, proj = _inputs(shape, h, 1 if m >= 14 else 3, 60 + m)
    V = torch.from_numpy(V).cuda()
    s = _solver(monkeypatch, "", shape, h, m, npl, pos, proj)
    chi, zeta = s.bounds(V, 24, 0.02)
    chi, zeta = chi.clone(), zeta.clone()
    mu = float(chi.median())
    some = torch.tensor([0, s.n_nodes - 1, 17, 17, 5, s.n_nodes // 2], dtype=torch.int64, device="cuda")
    for nodes in (None, some):
        out = {}
        for form in ("region", "", " "):
            if form.strip():
                monkeypatch.setenv("SQ_FORCE_KERNEL", form)
            else:
                monkeypatch.delenv("SQ_FORCE_KERNEL", raising=False)
            out[form] = s.nl_forces(V, mu, 0.1, chi=chi, zeta=zeta, nodes=nodes).clone()
        assert torch.equal(out[""], out[" "])
        scale = float(out["region"].abs().max())
        assert scale > 1e-6
        assert float((out[""] - out["region"]).abs().max()) <= 2 * FP32_FORCE * scale
    s.close()

"""Which form of the region kernels a context runs, as sq_context_info reports
it: the inputs of test_gpu_quad.py and test_gpu_quad_force.py run the quad
kernels where those tests compare them (Lanczos with projectors below 23^3 and
local regions below 17^3 keep the general kernels), and the general forms where
the environment or the precision asks for them."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_quad import GRIDS, _inputs, _solver  # noqa: E402


def _info(monkeypatch, kernel, m, nonlocal_, seed):
    from paper_1708_07913_gb300 import sq
    shape, h = GRIDS[m % 2], 0.5
    pos, _, proj = _inputs(shape, h, 1 if m >= 14 else 3, seed)
    s = _solver(monkeypatch, kernel, shape, h, m, 16, pos, proj if nonlocal_ else ())
    info = sq.sq_context_info(s.ctx)
    assert info["m"] == m
    return s, info


@pytest.mark.parametrize("nonlocal_", [False, True])
@pytest.mark.parametrize("m", range(6, 16))
def test_default_forms(monkeypatch, m, nonlocal_):
    from paper_1708_07913_gb300 import sq
    monkeypatch.delenv("SQ_FORCE_KERNEL", raising=False)
    for seed in (40 + m, 60 + m):                        # of the two files
        s, info = _info(monkeypatch, "", m, nonlocal_, seed)
        quad_mom = m >= (7 if nonlocal_ else 8)
        quad_lan = m >= (11 if nonlocal_ else 8)
        assert info["moments"] == (sq.FORM_QUAD if quad_mom else sq.FORM_GENERAL)
        assert info["lanczos"] == (sq.FORM_QUAD if quad_lan else sq.FORM_GENERAL)
        if not nonlocal_:
            assert info["forces"] == sq.FORM_NONE
        else:
            assert info["forces"] == (sq.FORM_QUAD if quad_mom else sq.FORM_GENERAL)
            for env, form in (("region", sq.FORM_GENERAL), ("legacy", sq.FORM_FIRST)):
                monkeypatch.setenv("SQ_FORCE_KERNEL", env)
                assert sq.sq_context_info(s.ctx)["forces"] == form
            monkeypatch.delenv("SQ_FORCE_KERNEL")
        s.close()


@pytest.mark.parametrize("kernel,form", [("cta", "FORM_GENERAL"), ("cluster", "FORM_CLUSTER")])
def test_forms_from_the_environment(monkeypatch, kernel, form):
    from paper_1708_07913_gb300 import sq
    s, info = _info(monkeypatch, kernel, 8, False, 48)
    assert info["moments"] == info["lanczos"] == getattr(sq, form)
    s.close()


def test_fp64_runs_the_general_forms(monkeypatch):
    from paper_1708_07913_gb300 import SQ_FP64, SQSolver, sq
    monkeypatch.delenv("SQ_FORCE_KERNEL", raising=False)
    pos, _, proj = _inputs(GRIDS[0], 0.5, 3, 48)
    s = SQSolver(GRIDS[0], 0.5, 4.1, 16, SQ_FP64, pos, proj)
    info = sq.sq_context_info(s.ctx)
    assert info["moments"] == info["lanczos"] == info["forces"] == sq.FORM_GENERAL
    s.close()

"""The warm-start network where its tiles end: axes of one node, of one less
and one more than a tile of the layers (16, 8, 4 and 2 nodes a side), and
several tiles along each axis; same weights, inputs and tolerances against
the FP64 oracle as in test_gpu_cnn.py."""
import numpy as np
import pytest

from oracle import cnn_oracle as cnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1708_07913_gb300 import build, sq  # noqa: E402
from test_gpu_cnn import DEV, _dev, _flat, _problem  # noqa: E402

build()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("shape", [(17, 3, 1), (1, 17, 5), (2, 1, 33), (15, 9, 4), (33, 18, 3), (7, 31, 9)])
def test_ragged_tiles_match_oracle(shape, bf16):
    p, V, ref = _problem(shape, seed=100 + sum(shape))
    net = sq.sq_cnn_create(32, bf16)
    sq.sq_cnn_set_params(net, _flat(p), p["v_shift"], p["v_scale"], p["rho_scale"])
    rho = torch.empty(V.size, dtype=torch.float64, device=DEV)
    sq.sq_cnn_forward(net, shape, _dev(V), rho)
    rho_o, _ = cnn.forward(p, V, bf16=bf16)
    np.testing.assert_allclose(rho.cpu().numpy(), rho_o.ravel(), rtol=0, atol=(2e-3 if bf16 else 1e-5) * np.abs(rho_o).max())
    L = sq.sq_cnn_backward(net, shape, _dev(V), _dev(ref), rho)
    L_o, g_o = cnn.backward(p, V, ref, bf16=bf16)
    assert abs(L - L_o) <= (1e-3 if bf16 else 1e-6) * L_o
    g = sq.sq_cnn_get_grads(net)
    off = 0
    for k in cnn.TRAINED:
        n = g_o[k].size
        a, b = g[off:off + n], g_o[k].ravel()
        off += n
        if bf16:
            assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b), k
        else:
            np.testing.assert_allclose(a, b, rtol=0, atol=1e-5 * np.abs(b).max(), err_msg=k)
    sq.sq_cnn_destroy(net)

"""Weight gradients of the warm-start network on a large grid.

On a constant field with a constant reference every node contributes the same,
so the gradient of the mean loss does not depend on the grid: 128^3 nodes are
held to the oracle on one node.  Equal terms of one sign are the hardest sums
for a serial FP32 chain, whose roundings then all go the same way.

Tolerance.  1e-5 of each tensor's largest entry for the network's FP32
arithmetic (test_gpu_cnn.py), and the roundings of the sum over the nodes: 128
of a tile's nodes one after another, 171 tiles of one block, 96 blocks, each at
most 2^-24 of the result."""
import numpy as np
import pytest

from oracle import cnn_oracle as cnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_cnn import DEV, _flat, _problem, sq  # noqa: E402

TOL = 1e-5 + (128 + 171 + 96) * 2.0 ** -24


@pytest.mark.parametrize("seed", [11, 12, 13])
def test_constant_field_gradient_does_not_depend_on_the_grid(seed):
    p, V, ref = _problem((1, 1, 1), seed)
    _, g_o = cnn.backward(p, V, ref)
    net = sq.sq_cnn_create(32, False)
    sq.sq_cnn_set_params(net, _flat(p), p["v_shift"], p["v_scale"], p["rho_scale"])
    n = 128
    full = lambda v: torch.full((n ** 3,), float(v.ravel()[0]), dtype=torch.float64, device=DEV)
    rho = torch.empty(n ** 3, dtype=torch.float64, device=DEV)
    sq.sq_cnn_backward(net, (n, n, n), full(V), full(ref), rho)
    g = sq.sq_cnn_get_grads(net)
    sq.sq_cnn_destroy(net)
    off = 0
    for k in cnn.TRAINED:
        b = g_o[k].ravel()
        np.testing.assert_allclose(g[off:off + b.size], b, rtol=0, atol=TOL * np.abs(b).max(), err_msg=k)
        off += b.size

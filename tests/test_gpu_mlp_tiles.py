"""Training kernels of the network at the edges of their tiles, against the FP64 oracle (needs a GB300).

128 batch rows, 64 or 32 columns and k-tiles of 64 per tile: batches around 64 and
128, widths that are no multiple of 4 (scalar loads and stores), one input, one
output. The bounds are those of test_gpu_learned.py for BF16 operands.
"""
import numpy as np
import pytest

from oracle import mlp as omlp
from tests.test_gpu_learned import DEV, _per_tensor, lib

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(13, 256, 12, b) for b in (1, 63, 64, 65, 127, 129, 4097)] + \
        [(56, 256, 55, 200), (1, 64, 1, 130), (5, 33, 7, 300), (130, 70, 66, 257)]


@pytest.mark.parametrize("n_in,hidden,n_out,B", CASES)
def test_gradients_at_tile_edges(n_in, hidden, n_out, B):
    shapes = omlp.layer_shapes(n_in, hidden, n_out)
    rng = np.random.default_rng(B)
    theta = omlp.init_params(n_in, hidden, n_out, seed=5) + rng.normal(0, 0.02, omlp.n_params(n_in, hidden, n_out))
    theta = theta.astype(np.float32).astype(np.float64)
    X, Y = (rng.normal(size=(B, n)).astype(np.float32) for n in (n_in, n_out))
    loss_ref, g_ref = omlp.loss_and_grad(theta, X.astype(np.float64), Y.astype(np.float64), shapes)
    net = lib().MLP(n_in, hidden, n_out)
    net.set_params(torch.tensor(theta.astype(np.float32), device=DEV))
    g = torch.full((net.nparams,), float("nan"), dtype=torch.float32, device=DEV)
    loss = torch.zeros(1, dtype=torch.float32, device=DEV)
    net.grad(torch.tensor(X, device=DEV), torch.tensor(Y, device=DEV), grad=g, loss=loss)
    torch.cuda.synchronize()
    assert abs(float(loss.item()) - loss_ref) <= 2e-2 * loss_ref
    for gg, gr in zip(_per_tensor(g.cpu().numpy().astype(np.float64), shapes), _per_tensor(g_ref, shapes)):
        assert np.linalg.norm(gg - gr) <= 2e-2 * np.linalg.norm(gr)

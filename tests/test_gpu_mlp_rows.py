"""Network gradients and forward passes at the edges of the row tiles: 128 rows in the layers and in the weight
gradients of narrow layers (at most 16 wide), 32 rows in the other weight gradients, and several tiles a block."""
import numpy as np
import pytest

from gpu_util import need_gpu, torch
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 32, 33, 127, 128, 129, 40001])
@pytest.mark.parametrize("n_in,width,depth,n_out", [(1, 1, 1, 1), (8, 3, 1, 3), (16, 16, 2, 16), (8, 17, 1, 3), (8, 33, 2, 3),
                                                    (128, 128, 2, 128)])
def test_rows(n, n_in, width, depth, n_out):
    """Against the FP64 oracle: sums of at most 128 products in FP32 (forward 1e-5), and over the rows besides
    (gradient 1e-4).  40,001 rows are several tiles for every block of every kernel."""
    tam = need_gpu()
    net = tam.Mlp(n_in, width, depth, n_out, seed=7)
    shapes = omlp.layer_shapes(n_in, width, depth, n_out)
    rng = np.random.default_rng(n)
    shift, scale = rng.standard_normal(n_in).astype(np.float32) * 0.1, (1.0 + rng.random(n_in)).astype(np.float32)
    out_scale = (0.5 + rng.random(n_out)).astype(np.float32)
    net.set_normalization(shift, scale, out_scale)
    theta = net.get_params().astype(np.float64)
    X, Y = rng.standard_normal((n, n_in)).astype(np.float32), rng.standard_normal((n, n_out)).astype(np.float32)
    args = (shift.astype(np.float64), scale.astype(np.float64), out_scale.astype(np.float64))
    ref, _ = omlp.forward(theta, shapes, X.astype(np.float64), *args)
    got = net.forward(torch.from_numpy(X).cuda()).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max() + 1e-6
    loss_o, g_o = omlp.loss_and_grad(theta, shapes, X.astype(np.float64), Y.astype(np.float64), *args)
    loss, g = net.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    assert abs(loss - loss_o) <= 1e-5 * loss_o
    assert np.linalg.norm(g - g_o) <= 1e-4 * np.linalg.norm(g_o)

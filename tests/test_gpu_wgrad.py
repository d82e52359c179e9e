"""Weight and bias gradients of the network where a CTA sums several tiles: at
these sizes the layers have more 16 x 16 tiles than groups of tiles (at 64 x 64
every group is one tile), with remainders and unequal numbers of tiles per row
and column."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import unet  # noqa: E402
from paper_1802_03770_gb300.api import Net  # noqa: E402
from tests.test_gpu_unet import _layer_input, unflatten  # noqa: E402


@pytest.mark.parametrize("H,W", [(320, 448), (448, 192)])
@pytest.mark.parametrize("tensor_cores", [False, True])
def test_weight_gradients_of_tile_groups(H, W, tensor_cores):
    """Layer by layer from the GPU's own activations and upstream gradients: FP32
    sums against FP64 ones, relative 2-norm <= 1e-4 as at 64 x 64 (a tile left
    out or taken twice costs >= 1e-2)."""
    net = Net(H, W, seed=21)
    net.tensor_cores(tensor_cores)
    params = unflatten(net.get_params())
    rng = np.random.default_rng(22)
    xs = torch.tensor(rng.standard_normal((1, 3, H, W)), dtype=torch.float32, device="cuda:0")
    ts = torch.tensor(rng.standard_normal((1, 1, H, W)), dtype=torch.float32, device="cuda:0")
    net.loss_grad(xs, ts)
    net.check()
    acts = [net.get_tensor(i).astype(np.float64) for i in range(12)]
    grads = [net.get_tensor(i, grad=True).astype(np.float64) for i in range(12)]
    _, g = net.get_params(grads=True)
    i = 0
    for li, name in enumerate(unet.LAYERS):
        w, b = params[name]
        gz = grads[li + 1] * (acts[li + 1] > 0) if name != "head" else grads[li + 1]
        _, dw, db = unet.conv_backward(_layer_input(acts, name), w, gz)
        for part, ref in ((g[i:i + w.size], dw), (g[i + w.size:i + w.size + b.size], db)):
            assert np.linalg.norm(part - ref.ravel()) <= 1e-4 * np.linalg.norm(ref), name
        i += w.size + b.size

"""The network's training step at the smallest and at uneven sizes: one image
and several, one and three 128-pixel strips per row, so that a weight-gradient
block's rows end inside, at and across a strip's last row. Gradients against
the FP64 reference with the GPU's BF16 storage points (as in test_gpu_net)."""
import numpy as np
import pytest

from oracle import net as ON
from gpu_util import rel_l2
from test_gpu_net import _inputs, _theta, grad_bf16

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n", [(1, 128), (3, 128), (7, 128), (1, 384)])
def test_gradient_shapes(B, n):
    from paper_1610_05258_gb300 import Net
    x, t = _inputs(B, n, 10 + B)
    theta = _theta(5)
    net = Net(n, B)
    net.load(theta)
    net.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), lr=0.0)
    g = net.grad()
    want = sum(grad_bf16(theta.astype(np.float64), x[b], t[b])[0] for b in range(B)) / B
    offs = np.cumsum([0] + [int(np.prod(s)) for s in ON.param_shapes()])
    for k in range(8):
        # BF16 flips of stored activations between FP32 and FP64 sums: below
        # 1e-3 of a block's gradient (2^-9 of the few values that flip)
        assert rel_l2(g[offs[k]:offs[k + 1]], want[offs[k]:offs[k + 1]]) <= 1e-3, k

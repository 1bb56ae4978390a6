"""A network with a layer whose weight gradient alone is larger than the scratch
of split partials (2048 x 18432 weights at the coarsest of six levels): a
training step on a batch follows the sum of the samples' own gradients.

The first Adam step is -lr g / (|g| + eps); the gradients of both sides differ
by the rounding of dy to bfloat16 at most (2^-8 of a term), which moves the
step of an entry above 1e-2 of the layer's largest by less than 1e-2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402
from paper_2009_12663_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_batch_step_of_a_layer_wider_than_the_scratch():
    batch, H, W, lr = 2, 32, 256, 1e-3
    net = gb.Unet(levels=6, base=64, cin=5, cout=3, height=H, width=W)
    net.set_params(torch.tensor(learned.he_init(net, 3), device=DEV))
    rng = np.random.default_rng(5)
    x = torch.tensor(rng.standard_normal((batch, 5, H, W)).astype(np.float32), device=DEV)
    t = torch.tensor(rng.standard_normal((batch, 3, H, W)).astype(np.float32), device=DEV)
    total = torch.zeros(net.num_params, device=DEV)
    for b in range(batch):
        y, g = torch.zeros(3, H, W, device=DEV), torch.zeros(net.num_params, device=DEV)
        net.forward(x[b].contiguous(), y)
        net.gradient(x[b].contiguous(), (2.0 * (y - t[b]) / (y.numel() * batch)).contiguous(), g)
        total += g
    p0, p1 = torch.zeros(net.num_params, device=DEV), torch.zeros(net.num_params, device=DEV)
    net.get_params(p0)
    net.train_step(x, t, lr)
    net.get_params(p1)
    step, wide = p1 - p0, 0
    for co, ci, k, coutp, kcp, wo, bo in net.layers():
        g, d = total[wo:wo + coutp * kcp], step[wo:wo + coutp * kcp]
        big = g.abs() > 1e-2 * g.abs().max()
        assert int(big.sum()) > 10
        assert torch.allclose(d[big], -lr * g[big] / (g[big].abs() + 1e-8), rtol=1e-2, atol=1e-6), (co, ci)
        wide += coutp * kcp > 32 << 20
    assert wide

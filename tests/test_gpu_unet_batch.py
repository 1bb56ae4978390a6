"""A training step on a batch against the sum of the samples' own gradients
(gbfwi_unet_gradient), at sizes on both sides of the kernels' choices: a tap a
block or nine in one, few weight gradients with many partials and many with
few, one sample and several, one level and four.

The first Adam step is -lr g / (|g| + eps), the sign of the gradient where it
is far above eps; the loss is the mean of the samples' in FP64 from FP32
outputs (1e-5, as for a single sample).  The gradients the two sides form
differ by the rounding of dy to bfloat16 at most (2^-8 of a term), far below
what could turn the sign of an entry above 1e-2 of the largest."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402
from paper_2009_12663_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("levels,base,H,W,batch", [(1, 8, 8, 64, 3), (3, 32, 24, 64, 1), (3, 32, 24, 64, 5), (4, 16, 32, 128, 9),
                                                   (4, 32, 64, 256, 2)])
def test_batch_step_sums_the_samples(levels, base, H, W, batch):
    net = gb.Unet(levels=levels, base=base, cin=5, cout=3, height=H, width=W)
    net.set_params(torch.tensor(learned.he_init(net, 3), device=DEV))
    rng = np.random.default_rng(levels + batch)
    x = torch.tensor(rng.standard_normal((batch, 5, H, W)).astype(np.float32), device=DEV)
    t = torch.tensor(rng.standard_normal((batch, 3, H, W)).astype(np.float32), device=DEV)
    total = torch.zeros(net.num_params, device=DEV, dtype=torch.float64)
    losses = []
    for b in range(batch):
        y, g = torch.zeros(3, H, W, device=DEV), torch.zeros(net.num_params, device=DEV)
        net.forward(x[b].contiguous(), y)
        losses.append(float(((y.double() - t[b].double()) ** 2).mean()))
        net.gradient(x[b].contiguous(), (2.0 * (y - t[b]) / (y.numel() * batch)).contiguous(), g)
        total += g.double()
    p0, p1 = torch.zeros(net.num_params, device=DEV), torch.zeros(net.num_params, device=DEV)
    net.get_params(p0)
    lr = 1e-3
    loss = net.train_step(x, t, lr)
    net.get_params(p1)
    assert abs(loss - np.mean(losses)) <= 1e-5 * np.mean(losses)
    step, gv = (p1 - p0).cpu().numpy(), total.cpu().numpy()
    big = np.abs(gv) > 1e-2 * np.abs(gv).max()
    assert big.sum() > 10
    assert np.allclose(step[big], -lr * np.sign(gv[big]), rtol=1e-2, atol=1e-6)

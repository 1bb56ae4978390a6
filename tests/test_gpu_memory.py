"""Calls that prefer more shots at once than their schedule asks for, with little
device memory left: the schedule's own batch is used, with the same results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402
from paper_2009_12663_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H, DT, NT, NSHOT, NREC = 25.0, 5e-4, 400, 24, 2000
LEFT = 160 << 20               # a shot's levels take 43 MB and its records 6 MB; all shots' 1 GB and 154 MB


def mesh():
    L = 40 * H
    src = [dict(x=L * (i + 0.5) / NSHOT, z=10.0, type=0, f0=15.0, t0=0.05, amp=1e12) for i in range(NSHOT)]
    m = gb.Mesh(40, 20, H, DT, NT, src, np.stack([np.linspace(0.0, L, NREC), np.zeros(NREC)], axis=1))
    x, z = (torch.tensor(a, device=DEV) for a in m.node_coords())
    vp = 2600.0 + 300.0 * torch.sin(x / 300.0) + 0.2 * z
    m.set_model(*(a.float().contiguous() for a in (2000.0 + 0.01 * x, vp, vp / 1.8)))
    return m


def fill(left=LEFT):
    """Device memory taken until `left` bytes are free."""
    held = []
    torch.cuda.empty_cache()
    while True:
        free = torch.cuda.mem_get_info()[0]
        if free <= left + (4 << 20):
            return held
        held.append(torch.empty(min(free - left, 8 << 30), dtype=torch.uint8, device=DEV))


def test_a_schedule_that_fits_runs_when_memory_is_short():
    ids = list(range(NSHOT))
    obs = torch.zeros(NSHOT, NREC, 2, NT, device=DEV)

    def call(m, g, H_, B0):
        f = m.misfit(ids, obs)
        f2 = m.adjoint_gradient(ids, obs, g)
        m.precond_diag(ids, 3, 50.0, 1.0, H_, B0)
        return f, f2

    a, b = ([torch.zeros(3, 81, 161, device=DEV) for _ in range(3)] for _ in range(2))
    want = call(mesh(), *a)                              # (the mesh gives its buffers back)
    m = mesh()
    held = fill()
    try:
        got = call(m, *b)
    finally:
        del held
        torch.cuda.empty_cache()
    assert got == want and torch.equal(a[0], b[0])
    # the map by steps instead of from levels: sums of NT non-negative terms in another order
    for c in range(3):
        assert (a[1][c] - b[1][c]).abs().max() <= 2 * NT * 2.0 ** -24 * a[1][c].max()


def test_training_takes_fewer_samples_at_once_when_memory_is_short():
    """Samples add to the gradients in order, however many are taken at once; a
    failed step leaves the network able to go on."""
    batch, Hn, Wn = 64, 32, 128
    gen = torch.Generator(device=DEV).manual_seed(4)
    x = torch.randn(batch, 5, Hn, Wn, generator=gen, device=DEV)
    t = torch.randn(batch, 3, Hn, Wn, generator=gen, device=DEV)

    def network():
        net = gb.Unet(levels=4, base=32, cin=5, cout=3, height=Hn, width=Wn)
        net.set_params(torch.tensor(learned.he_init(net, 1), device=DEV))
        return net
    net = network()
    p, q = torch.zeros(net.num_params, device=DEV), torch.zeros(net.num_params, device=DEV)
    y, y2 = torch.zeros(3, Hn, Wn, device=DEV), torch.zeros(3, Hn, Wn, device=DEV)
    losses = [net.train_step(x, t, 1e-3) for _ in range(2)]
    net.get_params(p)
    net.forward(x[0].contiguous(), y)
    del net
    net, x0 = network(), x[0].contiguous()
    held = fill(96 << 20)                                # all 64 samples' buffers take some 400 MB
    try:
        again = [net.train_step(x, t, 1e-3) for _ in range(2)]
        net.forward(x0, y2)
    finally:
        del held
        torch.cuda.empty_cache()
    net.get_params(q)
    assert again == losses and torch.equal(p, q) and torch.equal(y, y2)

"""Calls that prefer more shots at once than their schedule asks for, with little
device memory left: the schedule's own batch is used, with the same results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

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


def fill():
    """Device memory taken until LEFT bytes are free."""
    held = []
    torch.cuda.empty_cache()
    while True:
        free = torch.cuda.mem_get_info()[0]
        if free <= LEFT + (4 << 20):
            return held
        held.append(torch.empty(min(free - LEFT, 8 << 30), dtype=torch.uint8, device=DEV))


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

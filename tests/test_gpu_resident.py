"""The two forms of the time loop give the same results: the resident loop
(sem_resident.cu; meshes whose fields fit the SMs) and one kernel per step
(sem_step.cu; larger meshes).

A disturbance travels at most one element per step, so the records of a mesh
that fits and of a 700 x 80 element one that does not, sharing the top left
corner, the model and the acquisition, agree until the far edges of the
smaller one are reached: bitwise for the fields (same element arithmetic,
same order of every sum).  The strain sums of the gradient are summed over
time by element in one form and by node in the other: nt additions of FP32
values in another order, nt 2^-24 of the largest entry per parameter (nt <=
15: 1e-6; asserted 4e-6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H, DT = 25.0, 5e-4


def simulate(nex, nez, top, nt, src, rec, **sched):
    m = gb.Mesh(nex, nez, H, DT, nt, src, rec, free_surface_top=top)
    m.set_schedule(**sched)
    x, z = (torch.tensor(a, device=DEV) for a in m.node_coords())
    vp = 2600.0 + 300.0 * torch.sin(x / 90.0) + 0.2 * z
    m.set_model(*(a.float().contiguous() for a in (2000.0 + 0.1 * x, vp, vp / 1.8)))
    obs = torch.zeros(len(src), len(rec), 2, nt, device=DEV)
    ids = list(range(len(src)))
    seis = m.forward(ids, torch.zeros_like(obs)).clone()
    f = m.misfit(ids, obs)
    grad = torch.zeros(3, m.nz, m.nx, device=DEV)
    assert m.adjoint_gradient(ids, obs, grad) == f
    return seis, f, grad


# tiles of one CTA and of several, ragged last tiles, one element past a full tile
@pytest.mark.parametrize("nex,nez,top", [(16, 15, 1), (19, 16, 0), (33, 17, 1), (37, 20, 1), (64, 31, 0)])
@pytest.mark.parametrize("sched", [dict(), dict(shots_per_launch=2, ckpt_every=4)])
def test_resident_loop_equals_step_kernels(nex, nez, top, sched):
    # sources (and every receiver) at least nt + 1 elements from the right and lower edges
    src = [dict(x=0.9 * H, z=0.4 * H, type=0, f0=40.0, t0=0.002, amp=1e9),
           dict(x=2.0 * H, z=1.3 * H, type=2, f0=40.0, t0=0.002, amp=1e9)]
    rec = np.array([[0.0, 0.0], [H, 0.0], [1.7 * H, 0.3 * H], [2.0 * H, 2.0 * H], [0.2 * H, 2.9 * H]])
    nt = min(nex, nez) - 4
    nt = min(nt, 15)
    a = simulate(nex, nez, top, nt, src, rec, **sched)
    b = simulate(700, 80, top, nt, src, rec, **sched)
    assert a[0].abs().max() > 0
    assert torch.equal(a[0], b[0])
    assert abs(a[1] - b[1]) <= 1e-12 * abs(b[1])
    nz, nx = 4 * (nez - 1), 4 * (nex - 1)                 # nodes whose mass and moduli sums agree
    for c in range(3):
        d = (a[2][c, :nz, :nx] - b[2][c, :nz, :nx]).abs().max()
        assert d <= 4e-6 * b[2][c].abs().max(), (c, float(d))

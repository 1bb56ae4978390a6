"""The raw preconditioner maps from stored levels (meshes whose time loop is
resident, sem_integrals.cu) equal those of the preconditioner steps
(sem_step.cu) on a mesh too large for it that shares the top left corner.

The levels and a step's terms are bitwise the same; the sums of nt terms run
by element or node instead of by step: nt 2^-24 of the largest entry, below
2e-6 with nt <= 15 and the elements around a node (asserted 8e-6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H, DT = 25.0, 5e-4


def raw_map(nex, nez, top, nt, src, rec, kind, **sched):
    m = gb.Mesh(nex, nez, H, DT, nt, src, rec, free_surface_top=top)
    m.set_schedule(**sched)
    x, z = (torch.tensor(a, device=DEV) for a in m.node_coords())
    vp = 2600.0 + 300.0 * torch.sin(x / 90.0) + 0.2 * z
    m.set_model(*(a.float().contiguous() for a in (2000.0 + 0.1 * x, vp, vp / 1.8)))
    raw, B0 = torch.zeros(3, m.nz, m.nx, device=DEV), torch.zeros(3, m.nz, m.nx, device=DEV)
    m.precond_diag(list(range(len(src))), kind, 50.0, 1.0, raw, B0)
    return raw


# one tile and several, ragged last tiles; all shots together and in batches; checkpoints
@pytest.mark.parametrize("nex,nez,top,sched", [(16, 15, 1, dict()), (19, 16, 0, dict(shots_per_launch=2)),
                                               (37, 20, 1, dict(ckpt_every=4)), (64, 31, 0, dict(streams=2))])
@pytest.mark.parametrize("kind", [1, 2, 3, 4])
def test_maps_from_levels_equal_preconditioner_steps(nex, nez, top, sched, kind):
    src = [dict(x=(0.9 + 0.4 * i) * H, z=(0.4 + 0.3 * i) * H, type=i % 3, f0=40.0, t0=0.002, amp=1e9) for i in range(3)]
    rec = np.array([[0.0, 0.0], [H, 0.0], [1.7 * H, 0.3 * H], [2.0 * H, 2.0 * H], [0.2 * H, 2.9 * H]])
    nt = min(min(nex, nez) - 5, 15)
    a = raw_map(nex, nez, top, nt, src, rec, kind, **sched)
    b = raw_map(700, 80, top, nt, src, rec, kind, **sched)
    nz, nx = 4 * (nez - 1), 4 * (nex - 1)                # nodes whose element sums agree
    for c in range(3):
        assert a[c].abs().max() > 0
        d = (a[c, :nz, :nx] - b[c, :nz, :nx]).abs().max()
        assert d <= 8e-6 * b[c, :nz, :nx].abs().max(), (c, float(d))

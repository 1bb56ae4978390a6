"""Calls that take their shots in several batches, the last of them smaller,
against the same shots in other batches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H, DT = 50.0, 5e-4


def mesh(nex, nez, nt, nshot, nrec=29, same=False, **sched):
    """Shots along the surface, or all at one place."""
    L = nex * H
    src = [dict(x=L * (0.5 if same else (i + 0.5) / nshot), z=20.0, type=0, f0=8.0, t0=0.05, amp=1e12) for i in range(nshot)]
    rec = np.stack([np.linspace(0.0, L, nrec), np.zeros(nrec)], axis=1)
    m = gb.Mesh(nex, nez, H, DT, nt, src, rec)
    m.set_schedule(**sched)
    x, z = (torch.tensor(a, device=DEV) for a in m.node_coords())
    vp = 2600.0 + 300.0 * torch.sin(x / 900.0) + 0.2 * z
    m.set_model(*(a.float().contiguous() for a in (2000.0 + 0.01 * x, vp, vp / 1.8)))
    return m


def raw_map(m, ids, kind):
    raw, B0 = (torch.zeros(3, m.nz, m.nx, device=DEV) for _ in range(2))
    m.precond_diag(ids, kind, 100.0, 1.0, raw, B0)
    return raw


# Levels of 6 GiB hold three of these shots: batches of 3, .., 1 and 3, 2.  A
# forward map sums squares, so it is the sum of the shots' own maps (different
# shots).  A receiver map is the modulus of a sum: of equal shots it is nshot times
# one shot's.  The chunks of time are those of any batch, so both sides differ by the
# FP32 additions of the shots (nshot 2^-24) and the products of the maps' finish (8
# 2^-24 on each side); where a field has only just arrived, by roundings of denormals.
@pytest.mark.parametrize("nex,nez,nshot,nt,kind", [(126, 46, 13, 1333, 3), (160, 60, 5, 500, 4)])
def test_map_in_ragged_batches_is_the_sum_of_its_shots(nex, nez, nshot, nt, kind):
    m = mesh(nex, nez, nt, nshot, same=kind == 4)
    total = torch.zeros(3, m.nz, m.nx, device=DEV, dtype=torch.float64)
    whole = raw_map(m, list(range(nshot)), kind).double()   # first: no other call has grown the buffers
    for i in range(nshot):
        total += raw_map(m, [i], kind).double()
    assert whole.abs().max() > 0
    assert bool(((whole - total).abs() <= (nshot + 16) * 2.0 ** -24 * total + 1e-30 * total.max()).all())


# the last batch (19, 13 and 20 shots of 43, 37 and 44) takes more of them in one launch
# than the first of 24; 50 shots of a mesh of one tile
@pytest.mark.parametrize("nex,nez,nshot,spl", [(280, 10, 43, 24), (253, 24, 37, 24), (110, 37, 44, 24), (14, 8, 50, 3)])
def test_records_of_ragged_batches_are_those_of_single_shots(nex, nez, nshot, spl):
    nt, ids = 40, list(range(nshot))
    m = mesh(nex, nez, nt, nshot, shots_per_launch=spl)
    seis = torch.zeros(nshot, 29, 2, nt, device=DEV)
    obs = torch.zeros_like(seis)
    f = m.misfit(ids, obs)                               # first: no other call has grown the buffers
    m.forward(ids, seis)
    one, each = torch.zeros(1, 29, 2, nt, device=DEV), 0.0
    for i in ids:
        m.forward([i], one)
        assert torch.equal(one[0], seis[i]), i           # the fields do not depend on the batch
        each += m.misfit([i], obs[:1])
    assert f > 0 and abs(f - each) <= 1e-13 * nshot * f   # FP64 sums of the shots' misfits


def test_many_shot_counts_on_one_mesh():
    """A study with changing minibatches: every number of shots and kind of pass
    keeps its plan, and none loses it to the others."""
    nshot, nt = 40, 30
    m = mesh(23, 19, nt, nshot, shots_per_launch=2)
    seis, again = (torch.zeros(nshot, 29, 2, nt, device=DEV) for _ in range(2))
    m.forward(list(range(nshot)), seis)
    first = raw_map(m, [0, 1], 2)
    for k in range(1, nshot + 1):
        m.forward(list(range(k)), again[:k])
        assert torch.equal(again[:k], seis[:k]), k
        raw_map(m, list(range(k)), 1 + k % 2)
    assert torch.equal(raw_map(m, [0, 1], 2), first)


# Batches of 10 and 8 (10 and 3), the whole history or checkpoints.  FP32 sums over the shots
# and in the chain rule: nshot 2^-24 of the shots' moduli, and of each shot's largest
# entry times nt where its terms cancel; asserted twice that.
@pytest.mark.parametrize("nshot,spl,ckpt", [(18, 10, 0), (13, 10, 0), (18, 10, 100)])
def test_gradient_in_ragged_batches_is_the_sum_of_its_shots(nshot, spl, ckpt, nrec=29):
    nt, ids = 500, list(range(nshot))
    m = mesh(46, 42, nt, nshot, nrec=nrec, shots_per_launch=spl, ckpt_every=ckpt)
    obs = torch.zeros(nshot, nrec, 2, nt, device=DEV)
    grad, one = (torch.zeros(3, m.nz, m.nx, device=DEV) for _ in range(2))
    f = m.adjoint_gradient(ids, obs, grad)
    total, size, each = torch.zeros_like(grad).double(), torch.zeros_like(grad).double(), 0.0
    for i in ids:
        each += m.adjoint_gradient([i], obs[:1], one)
        total += one
        size += one.abs() + nt * one.abs().amax(dim=(1, 2), keepdim=True)
    assert f > 0 and abs(f - each) <= 1e-13 * nshot * f
    assert bool(((grad - total).abs() <= 2 * nshot * 2.0 ** -24 * size).all())
    m.set_schedule(shots_per_launch=3, streams=2)        # gradients do not depend on the schedule
    m.adjoint_gradient(ids, obs, one)
    assert torch.equal(grad, one)


# Many receivers: a tile's lists take its shared memory, and the best tile for some numbers
# of shots no longer fits while that of others does (18 shots by 10 and 2000
# receivers: 8 shots); the next best one takes its place.
@pytest.mark.parametrize("nrec", [1000, 2000, 3000])
@pytest.mark.parametrize("nshot", [13, 18])
def test_gradient_where_a_batch_does_not_fit(nrec, nshot):
    test_gradient_in_ragged_batches_is_the_sum_of_its_shots(nshot, 10, 0, nrec)


@pytest.mark.parametrize("nrec", [2000, 6000, 12000])
def test_records_where_a_batch_does_not_fit(nrec):
    nt, nshot = 20, 23
    m = mesh(46, 42, nt, nshot, nrec=nrec, shots_per_launch=9)
    seis, one = torch.zeros(nshot, nrec, 2, nt, device=DEV), torch.zeros(1, nrec, 2, nt, device=DEV)
    m.forward(list(range(nshot)), seis)
    for i in range(nshot):
        m.forward([i], one)
        assert torch.equal(one[0], seis[i]), i
    for kind in (1, 2):
        assert bool(torch.isfinite(raw_map(m, list(range(nshot)), kind)).all())


def test_more_shots_than_a_grid_has_rows():
    """70000 shots of the smallest kind fit the memory a call takes beyond its
    schedule, but not one launch.  All equal: each gives the first one's part."""
    nshot, nt = 70000, 2
    m = mesh(5, 3, nt, nshot, nrec=2, same=True, shots_per_launch=2, streams=2)
    ids = list(range(nshot))
    obs = torch.ones(nshot, 2, 2, nt, device=DEV)
    grad, one = (torch.zeros(3, m.nz, m.nx, device=DEV) for _ in range(2))
    f1 = m.adjoint_gradient([0], obs[:1], one)
    f = m.adjoint_gradient(ids, obs, grad)
    assert f1 > 0 and abs(f - nshot * f1) <= 1e-15 * nshot * f    # one FP64 addition a shot
    assert abs(m.misfit(ids, obs) - f) <= 1e-15 * nshot * f
    # one FP32 addition a shot (their error grows like the number of equal terms: nshot 2^-24)
    assert (grad - nshot * one).abs().max() <= nshot * 2.0 ** -24 * nshot * one.abs().max()
    for kind in (1, 2):
        raw, first = raw_map(m, ids, kind), raw_map(m, [0], kind)
        assert (raw - nshot * first).abs().max() <= nshot * 2.0 ** -24 * nshot * first.max()

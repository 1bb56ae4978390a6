"""gbfwi_set_model: the fault of the first faulty node decides the error, a
rejected model leaves the old one in place, host and device arrays (and a
mixture) set the same model."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def mesh(nex=9, nez=5):
    return gb.Mesh(nex, nez, 25.0, 5e-4, 60, [dict(x=60.0, z=10.0, f0=30.0, amp=1e9)], np.array([[110.0, 0.0], [20.0, 50.0]]))


def arrays(m, seed=0):
    r = np.random.default_rng(seed)
    vp = (2500.0 + 500.0 * r.random((m.nz, m.nx))).astype(np.float32)
    return [(2000.0 + 100.0 * r.random((m.nz, m.nx))).astype(np.float32), vp, (vp / 1.8).astype(np.float32)]


def seismograms(m):
    return m.forward([0], torch.zeros(1, 2, 2, 60, device=DEV)).clone()


def dev(a):
    return torch.tensor(a, device=DEV)


@pytest.mark.parametrize("first,then,name", [("nan", "vs", "ENONFINITE"), ("vs", "nan", "EINVAL"), ("rho", "inf", "EINVAL"),
                                             ("inf", "rho", "ENONFINITE"), ("vp", "cfl", "EINVAL"), ("cfl", "cfl", "ECFL")])
@pytest.mark.parametrize("where", [(0, 1), (5, -1)])
def test_first_fault_decides(first, then, name, where):
    m = mesh()
    good = arrays(m)
    m.set_model(*(dev(a) for a in good))
    before = seismograms(m)
    flat = [a.copy() for a in good]
    faults = dict(nan=(1, np.nan), inf=(0, np.inf), vs=(2, 0.0), rho=(0, -1.0), vp=(1, 10.0), cfl=(1, 9e4))
    for at, f in zip(where, (first, then)):
        c, v = faults[f]
        flat[c].reshape(-1)[at] = v
    for put in (dev, lambda a: a):
        with pytest.raises(gb.GbfwiError) as e:
            m.set_model(*(put(a) for a in flat))
        assert e.value.name == name
    assert torch.equal(seismograms(m), before)


@pytest.mark.parametrize("put", [(0, 0, 0), (1, 0, 1), (0, 1, 0)])
def test_host_and_device_arrays(put):
    m = mesh()
    a = arrays(m, 3)
    m.set_model(*(dev(v) for v in a))
    want = seismograms(m)
    m.set_model(*(dev(v) for v in arrays(m, 4)))
    assert not torch.equal(seismograms(m), want)
    m.set_model(*(dev(v) if p else v for v, p in zip(a, put)))
    assert torch.equal(seismograms(m), want)

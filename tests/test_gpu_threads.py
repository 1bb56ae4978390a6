"""Several host threads, each with handles and a stream of its own: plans and
launches of one do not disturb those of another.  Every thread makes its meshes
and stores anew, so that choosing a tile, allowing its shared memory and launching
interleave with the others'."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H, DT = 50.0, 5e-4


def sem_work(nex, nez):
    src = [dict(x=nex * H * (i + 0.5) / 3, z=20.0, type=0, f0=8.0, t0=0.05, amp=1e12) for i in range(3)]
    rec = np.stack([np.linspace(0.0, nex * H, 17), np.zeros(17)], axis=1)
    m = gb.Mesh(nex, nez, H, DT, 60, src, rec)
    one = torch.ones(m.nz, m.nx, device=DEV)
    m.set_model(2000.0 * one, 2600.0 * one, 1500.0 * one)
    obs = torch.zeros(3, 17, 2, 60, device=DEV)
    grad = torch.zeros(3, m.nz, m.nx, device=DEV)
    return torch.tensor([m.misfit([0, 1, 2], obs), m.adjoint_gradient([0, 1, 2], obs, grad)]), grad


def bfgs_work(n, k):
    g = torch.Generator(device=DEV).manual_seed(n)
    B0 = torch.rand(n, generator=g, device=DEV) + 0.5
    torch.cuda.current_stream().synchronize()            # creation takes no stream
    b = gb.Bfgs(n, k, B0)
    for _ in range(k):
        s = torch.randn(n, generator=g, device=DEV)
        b.update(s, 2.0 * s + 0.1 * torch.randn(n, generator=g, device=DEV))
    V, lam = torch.zeros(8, n, device=DEV), torch.zeros(8, dtype=torch.float64, device=DEV)
    b.lowrank_exact(8, eps_prior=1.0, V=V, lam=lam, std=torch.zeros(n, device=DEV))
    return lam, b.apply(V, torch.zeros_like(V), gamma=0.9)


JOBS = [(sem_work, (12, 6)), (sem_work, (40, 20)), (sem_work, (23, 31)), (bfgs_work, (1000, 20)), (bfgs_work, (700, 43))]


def test_threads_do_not_disturb_each_other():
    want = [f(*a) for f, a in JOBS]
    torch.cuda.synchronize()
    wrong = []

    def work(j):
        f, a = JOBS[j]
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for _ in range(8):
                    got = f(*a)
                    st.synchronize()
                    if not all(torch.equal(x, y) for x, y in zip(got, want[j])):
                        wrong.append((j, "other results"))
        except Exception as e:  # noqa: BLE001
            wrong.append((j, repr(e)))
    threads = [threading.Thread(target=work, args=(j,)) for j in range(len(JOBS))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong


def test_a_store_is_complete_when_it_is_created():
    """Creation takes no stream: work queued on another one must not overtake it,
    however busy the default stream is."""
    n, k = 5000, 6
    want = bfgs_work(n, k)
    torch.cuda.synchronize()
    busy = torch.zeros(4096, 4096, device=DEV)
    torch.matmul(busy, busy)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    for _ in range(40):
        torch.matmul(busy, busy)                         # some 50 ms on the default stream
    with torch.cuda.stream(st):
        got = bfgs_work(n, k)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))

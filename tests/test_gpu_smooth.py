"""Smoothing, median, damping and inversion of a raw map (precond_from_hessian)
and the mask channels of the network's features against the FP64 oracle, at
the sizes where their kernels change paths: a few rows or columns left over
from a block, windows of one node and of more taps than one shared chunk,
even and odd node counts of the median, ties, one and many mask points.

A smoothed value is a weighted mean of positive values (weights in FP32, up to
n taps a side): relative error below n 2^-24 + 2e-6 (the exponential), n <=
405 here: below 1e-5 with roundings that do not all add up; the weights left
out beyond 5 sigma change values between 1 and 3 by up to 5e-6.  The median is
one of the smoothed values.  Asserted 2e-5."""
import numpy as np
import pytest

from oracle import sem as osem
from oracle import unet as ou

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402
from paper_2009_12663_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H = 25.0


def mesh(nex, nez, src=None, rec=None):
    src = src or [dict(x=0.7 * H, z=0.3 * H, f0=20.0)]
    return gb.Mesh(nex, nez, H, 5e-4, 4, src, np.array([[0.0, 0.0]] if rec is None else rec))


@pytest.mark.parametrize("nex,nez,sigma,damp", [(1, 1, 3.0, 1.0), (7, 3, 1.0, 0.5), (31, 5, 41.3, 1.0), (32, 9, 397.0, 0.0),
                                                (100, 2, 487.0, 2.0), (3, 100, 487.0, 1.0)])
@pytest.mark.parametrize("ties", [False, True])
def test_smoothing_median_inversion(nex, nez, sigma, damp, ties):
    m = mesh(nex, nez)
    r = np.random.default_rng(nex + nez)
    raw = (r.integers(1, 3, (3, m.nz, m.nx)) if ties else 1.0 + 2.0 * r.random((3, m.nz, m.nx))).astype(np.float32)
    raw[1] *= 1e6
    st = osem.Setup(osem.Mesh(nex, nez, H), 5e-4, 4, np.array([[0.0, 0.0]]))
    _, want = osem.smooth_damp_invert(st, raw.astype(np.float64), sigma, damp)
    B0 = torch.zeros(3, m.nz, m.nx, device=DEV)
    m.precond_from_hessian(torch.tensor(raw, device=DEV), sigma, damp, B0)
    got = B0.cpu().numpy().astype(np.float64)
    for c in range(3):
        assert (np.abs(got[c] - want[c]) / want[c]).max() < 2e-5, c
    host = np.zeros_like(raw)
    m.precond_from_hessian(raw, sigma, damp, host)
    assert np.array_equal(host, B0.cpu().numpy())


# points on one line, scattered, on top of each other and outside every node line
@pytest.mark.parametrize("nsrc,nrec,scatter", [(1, 1, False), (3, 33, False), (5, 40, True), (2, 130, True)])
def test_mask_channels(nsrc, nrec, scatter):
    nex, nez = 21, 10
    r = np.random.default_rng(nsrc)
    W, D = nex * H, nez * H
    pts = lambda n: np.stack([r.uniform(0, W, n), r.uniform(0, D, n) if scatter else np.full(n, 0.37 * H)], 1)  # noqa: E731
    s, rec = pts(nsrc), pts(nrec)
    rec[-1] = rec[0]
    m = mesh(nex, nez, [dict(x=x, z=z, f0=20.0) for x, z in s], rec)
    x, z = m.node_coords()
    mdl = (2000.0 + 1000.0 * r.random((3, m.nz, m.nx))).astype(np.float32)
    f = learned.features(m, torch.tensor(mdl, device=DEV), 32, 64).cpu().numpy()
    node = ou.features(*mdl, x, z, [tuple(p) for p in s], [tuple(p) for p in rec], learned.MASK_SIGMA_M)
    ref = ou.resample_bilinear(node, 32, 64)
    for c in range(5):
        assert np.abs(f[c] - ref[c]).max() <= 1e-5 * np.abs(ref[c]).max(), c

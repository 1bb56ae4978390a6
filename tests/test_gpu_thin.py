"""The inverse-Hessian apply on one or two vectors (thin products and
combination) against the FP64 oracle, at the edges of its tiles: 4096-column
chunks, 4-column threads, groups of eight rows, vectors that start off a
16-byte boundary, host arrays.  FP64 small matrices, compensated sums, FP32
coefficients: 2^-24 times the cancellation between the 2k terms (below 100 for
these histories), 6e-6; asserted 1e-4 like the wider products (a wrong
index gives O(1))."""
import numpy as np
import pytest

import synth
from oracle import bfgs as ob

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def t32(a):
    return torch.tensor(np.asarray(a, np.float32), device=DEV)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def shifted(a, off):
    """The array on the device, `off` floats past an allocation's start."""
    buf = torch.zeros(a.size + off, device=DEV)
    buf[off:] = t32(a).reshape(-1)
    return buf[off:].reshape(a.shape)


@pytest.mark.parametrize("n,k", [(40, 1), (999, 3), (4095, 4), (4096, 5), (4097, 8), (12289, 17), (70001, 40)])
@pytest.mark.parametrize("p,off", [(1, 0), (1, 1), (2, 0), (2, 3)])
def test_apply_one_or_two_vectors(n, k, p, off):
    S, Y, B0 = synth.synthetic_history(7, n, k)
    b = gb.Bfgs(n, k + 2, t32(B0))
    for i in range(k):
        b.update(shifted(S[i], off), Y[i].astype(np.float32) if i % 2 else t32(Y[i]))
    X = synth.gaussian_block(3, p, n).astype(np.float32)
    ref = ob.probe_block(X.astype(np.float64), S.astype(np.float64), Y.astype(np.float64), B0.astype(np.float64))
    for minus in (True, False):
        want = ref if minus else ref + B0.astype(np.float64) * X
        Z = shifted(np.zeros((p, n), np.float32), off)
        b.apply(shifted(X, off), Z, 1.0, minus_B0=minus)
        assert rel(Z.cpu().numpy(), want) < 1e-4
        host = np.zeros((p, n), np.float32)
        b.apply(X, host, 1.0, minus_B0=minus)
        assert np.array_equal(host, Z.cpu().numpy())

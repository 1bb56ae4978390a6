"""The autotuner's estimate of a schedule's device memory covers both forms of
the gradient (the buffers that csrc/sem_driver.cu reserves for each)."""
import pytest

pytest.importorskip("torch")
from paper_2009_12663_gb300 import autotune  # noqa: E402


@pytest.mark.parametrize("nex,nez", [(5, 3), (40, 20), (340, 70)])
@pytest.mark.parametrize("nshot,spl,streams", [(24, 1, 4), (24, 24, 1), (18, 10, 1), (7, 2, 4), (1, 8, 8)])
@pytest.mark.parametrize("nt,ckpt", [(500, 0), (500, 100), (130, 400)])
def test_estimate_covers_both_forms(nex, nez, nshot, spl, streams, nt, ckpt):
    nx, nz, nrec = 4 * nex + 1, 4 * nez + 1, 41
    NP = nz * ((nx + 3) // 4 * 4)
    full = ckpt <= 0 or ckpt >= nt
    levels = nt + 2 if full else ckpt + 6 + 3 * -(-nt // ckpt)
    common = (nshot + 1) * 5 * NP * 4 + nshot * nrec * 2 * nt * 4

    def batches(shots):                                # levels, velocities and adjoint ring, records, sums
        return shots * (8 * NP * (levels + 5) + nrec * 2 * nt * 4 + 5 * NP * 4)
    steps = batches(min(spl, nshot)) * min(streams, -(-nshot // min(spl, nshot)))
    most = min(spl * streams, nshot)
    resident = batches(most) + most * (25 * 2 + 2) * 4 * nex * nez + 32 * NP * most
    assert autotune.schedule_bytes(nx, nz, nshot, nrec, nt, spl, streams, ckpt) == common + max(steps, resident)

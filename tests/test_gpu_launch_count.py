"""gbfwi_launch_count counts every kernel once."""
import pytest

torch = pytest.importorskip("torch")
import paper_2009_12663_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


def test_resampling_is_one_launch():
    x, y = torch.ones(3, 8, 8, device="cuda:0"), torch.zeros(3, 16, 16, device="cuda:0")
    before = gb.launch_count()
    gb.resample(x, y, op=0)
    assert gb.launch_count() - before == 1 and torch.equal(y, torch.ones_like(y))

"""The shared-atomic probe returns the rate it measured, not a rounded one, the same
at every call."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("same_address", [False, True])
def test_probe_reports_its_measurement(same_address):
    from paper_1208_3658_gb300 import wtheta as W
    v = [W.wtheta_probe_shared_atomics(same_address) for _ in range(4)]
    assert all(x != round(x, 3) for x in v)
    assert max(v) - min(v) <= 1e-5 * max(v)

"""The serving loop's workspace model: a round is charged what the library takes for it,
which is less an item in large calls than in small ones."""
import pytest

from paper_2501_03245_gb300 import serving


def test_the_largest_call_bounds_the_charge():
    srv = object.__new__(serving.Server)
    srv.model = {"verify": (0.0, 1640.0), "msm": (10e6, 272.0)}
    srv.top = {"verify": (1 << 18, 128e6, 0.0), "msm": (1 << 20, 182e6, 164.0)}
    slack = lambda b: int(1.25 * b) + (1 << 20)  # noqa: E731
    assert srv.cost("verify", 1000) == slack(1640e3)
    assert srv.cost("verify", 1 << 18) == slack(128e6)
    assert srv.cost("msm", 1 << 15) == slack(10e6 + 272.0 * (1 << 15))
    assert srv.cost("msm", 1 << 20) == slack(182e6)
    assert srv.cost("msm", 1 << 22) == slack(182e6 + 164.0 * 3 * (1 << 20))


@pytest.mark.gpu
def test_measured_charge_of_large_calls(gpu_lib):
    """2^18 triples: at least the 128 MB a full GPU of items holds, and no more than the
    slack above it (four times that by the slope of small rounds).  2^20 points on a table
    of 16-bit windows: 182 MB (295 by the slope)."""
    import torch

    srv = serving.Server(torch, pool_triples=1 << 18, n_bases=1 << 20, pool_scalars=1 << 20)
    try:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        full = sms * 4 * 128 * 1644
        assert 0.9 * full < srv.cost("verify", 1 << 18) < 1.3 * full + (2 << 20)
        assert 182e6 < srv.cost("msm", 1 << 20) < 1.3 * 182e6 + (2 << 20)
        assert srv.cost("verify", 4096) < srv.cost("verify", 1 << 16) <= srv.cost("verify", 1 << 18)
    finally:
        srv.close()

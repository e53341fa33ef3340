"""The serving loop's workspace model: a round is charged what the library takes for it,
which for verification stops growing at the items the GPU works on at once."""
import pytest

from paper_2501_03245_gb300 import serving


def test_verification_is_charged_up_to_its_largest_round():
    srv = object.__new__(serving.Server)
    srv.model = {"verify": (0.0, 1640.0), "msm": (1e6, 300.0)}
    srv.verify_top = 128 << 20
    assert srv.cost("verify", 1000) == int(1.25 * 1640e3) + (1 << 20)
    assert srv.cost("verify", 1 << 18) == int(1.25 * (128 << 20)) + (1 << 20)
    assert srv.cost("msm", 1 << 22) == int(1.25 * (1e6 + 300.0 * (1 << 22))) + (1 << 20)


@pytest.mark.gpu
def test_measured_charge_of_a_large_round(gpu_lib):
    """2^18 triples: at least the 128 MB a full GPU of items holds, and no more than the
    slack above it (four times that by the slope of small rounds)."""
    import torch

    srv = serving.Server(torch, pool_triples=1 << 18, n_bases=4096, pool_scalars=1 << 14)
    try:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        full = sms * 4 * 128 * 1644
        assert 0.9 * full < srv.cost("verify", 1 << 18) < 1.3 * full + (2 << 20)
        assert srv.cost("verify", 4096) < srv.cost("verify", 1 << 16) <= srv.cost("verify", 1 << 18)
    finally:
        srv.close()

"""The multiply-adds that the benchmark's fractions count for scalar multiplications in
registers: products by the shape of the prime, below the textbook's count."""
import pytest

from paper_2501_03245_gb300 import costmodel


def test_point_operations():
    assert costmodel._ladder_point_imad("P-256") == (4 * 64 + 4 * 36, 8 * 64 + 3 * 36)
    assert costmodel._ladder_point_imad("secp256k1") == (3 * 73 + 4 * 45, 8 * 73 + 3 * 45)


@pytest.mark.parametrize("curve", sorted(costmodel.LADDER_PRODUCT_IMAD))
def test_below_the_textbook(curve):
    dbl, add = costmodel._ladder_point_imad(curve)
    doublings = 126 if curve == "secp256k1" else 256
    v = costmodel.ladder_verify_imad(curve)
    assert doublings * dbl + 79 * add < v < 1.07 * (doublings * dbl + 80 * add)
    assert v < costmodel.verify_imad()
    m = costmodel.imad_per_modmul(8)
    assert 15 * add < costmodel.ladder_fpmul_imad(curve) < costmodel.fpmul_modmul() * m
    assert 30 * add < costmodel.ladder_sign_imad(curve) < costmodel.sign_modmul() * m

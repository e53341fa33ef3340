"""The batched affine accumulation, fold and reduction (calls of 12 Mi digits or more) on
exceptional inputs: equal points (every addition of a bucket a doubling), P and -P in
turn (sums that cancel), O among the points, most scalars equal, and sizes one point
below and above the line between the two forms.  Narrow windows bring a call of a few
hundred thousand points to that many digits.  Points are a_i G: the sum is
(sum k_i a_i) G."""
import numpy as np
import pytest

from oracle import curves, ec
from paper_2501_03245_gb300 import synth
from tests.helpers import from_cuda, limbs_to_points, to_cuda

pytestmark = pytest.mark.gpu
LINE = 12 << 20  # digits from which a call takes the affine form
HALF_BITS = 126  # a split BN254 scalar's halves


def _windows(cid, c):
    """Digits of a scalar: of both halves on BN254, whose scalars are split."""
    return 2 * ((HALF_BITS + c) // c) if cid == 2 else (255 + c) // c


def _multiples(lib, cid, a):
    import torch

    out = torch.empty((len(a), 2 * curves.BY_ID[cid].limbs), dtype=torch.int32, device="cuda")
    lib.ecc_fixed_base_mul(cid, len(a), to_cuda(synth.ints_to_limbs(a, 8)), out)
    return out


class Case:
    """n points on curve cid with c-bit windows in the size class of n."""

    def __init__(self, lib, cid, n, c):
        self.lib, self.cid, self.C, self.n, self.c = lib, cid, curves.BY_ID[cid], n, c

    def __enter__(self):
        self.lib.ecc_msm_set_window(self.cid, self.n.bit_length() - 1, self.c)
        return self

    def __exit__(self, *exc):
        self.lib.ecc_msm_set_window(self.cid, self.n.bit_length() - 1, 0)
        return False

    def check(self, pts, a, k):
        import torch

        C = self.C
        out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")
        kd = to_cuda(synth.ints_to_limbs(k, 8))
        self.lib.ecc_msm(self.cid, self.n, pts, kd, out)
        total = sum(x * y for x, y in zip(a, k)) % C.n
        want = ec.mul(C, total, C.G) if total else None
        assert limbs_to_points(C, from_cuda(out).view(np.uint32))[0] == want
        offs = to_cuda(np.array([0, self.n], np.int64))
        self.lib.ecc_msm_ragged_dev(self.cid, 1, self.n, offs, pts, kd, out.zero_(), self.c)
        assert limbs_to_points(C, from_cuda(out).view(np.uint32))[0] == want


def _ints(q, n, seed):
    raw = np.random.default_rng(seed).bytes(40 * n)
    return [int.from_bytes(raw[40 * i:40 * i + 40], "little") % q for i in range(n)]


@pytest.mark.parametrize("cid,c", [(2, 4), (2, 8), (3, 4), (3, 8)])
def test_exceptional_sums(gpu_lib, cid, c):
    C = curves.BY_ID[cid]
    n = LINE // _windows(cid, c) + 1000
    few = _ints(C.n, 7, 1)
    k0 = _ints(C.n, 1, 2)[0]
    same = [few[0]] * n
    turn = [few[0] if i & 1 else C.n - few[0] for i in range(n)]
    mix = [few[i % 7] if i % 5 else 0 for i in range(n)]  # O in every fifth row
    k_few = [few[(i * i) % 7] if i % 3 else k0 for i in range(n)]
    k_bits = [i * 2654435761 >> 7 & 1 for i in range(n)]
    with Case(gpu_lib, cid, n, c) as case:
        p = _multiples(gpu_lib, cid, [few[0]]).repeat(n, 1)
        case.check(p, same, [k0] * n)        # one bucket a window, all doublings
        case.check(p, same, [1] * n)
        case.check(p, same, k_few)
        p = _multiples(gpu_lib, cid, turn[:2]).repeat(n // 2 + 1, 1)[:n].contiguous()
        case.check(p, turn, [k0] * n)        # P and -P in one bucket
        case.check(p, turn, k_few)
        p = _multiples(gpu_lib, cid, mix[:35]).repeat(n // 35 + 1, 1)[:n].contiguous()
        case.check(p, mix, [k0] * n)
        case.check(p, mix, k_few)
        case.check(p, mix, k_bits)
        case.check(p, mix, [0] * (n - 1) + [k0])
        p.zero_()
        case.check(p, [0] * n, k_few)        # nothing but O


@pytest.mark.parametrize("cid,c", [(2, 6), (3, 6)])
def test_each_side_of_the_line(gpu_lib, cid, c):
    C = curves.BY_ID[cid]
    top = -(-LINE // _windows(cid, c))  # the first size of the affine form
    a, k = _ints(C.n, top + 1, 3), _ints(C.n, top + 1, 4)
    for i in range(0, top, 1000):
        a[i], k[i] = a[0], k[0]
    pts = _multiples(gpu_lib, cid, a)
    for n in (top - 1, top, top + 1):
        with Case(gpu_lib, cid, n, c) as case:
            case.check(pts[:n], a[:n], k[:n])


@pytest.mark.parametrize("cid", [2, 3])
def test_ragged_on_a_window_table(gpu_lib, cid):
    """Resident bases, equal and opposite ones among them, instances of every size from
    none to all, in one affine call."""
    import torch

    C, n, c = curves.BY_ID[cid], 5000, 16
    few = _ints(C.n, 3, 5)
    a = [few[i % 3] if i & 1 else C.n - few[i % 3] for i in range(n)]
    W = (C.n.bit_length() + c) // c
    sizes = [0, 1, 31, 32, 33, n] + [n] * (LINE // (W * n) + 1)
    total = sum(sizes)
    k_few = _ints(C.n, 4, 6)
    k = [k_few[i * 7919 % 4] if i % 11 else 0 for i in range(total)]
    kd = to_cuda(synth.ints_to_limbs(k_few + [0], 8)[[i * 7919 % 4 if i % 11 else 4 for i in range(total)]])
    want, lo = [], 0
    for s in sizes:
        t = sum(x * y for x, y in zip(a, k[lo:lo + s])) % C.n
        want.append(ec.mul(C, t, C.G) if t else None)
        lo += s
    out = torch.zeros((len(sizes), 2 * C.limbs), dtype=torch.int32, device="cuda")
    h = gpu_lib.ecc_bases_create(cid, n, _multiples(gpu_lib, cid, a))
    try:
        gpu_lib.ecc_bases_precompute(h, c)
        gpu_lib.ecc_msm_bases_ragged(h, len(sizes), np.array(sizes, np.uint64), kd, out)
        assert limbs_to_points(C, from_cuda(out).view(np.uint32)) == want
        gpu_lib.ecc_msm_bases_ragged_dev(h, len(sizes), total, to_cuda(np.array(sizes, np.int64)), kd, out.zero_())
        assert limbs_to_points(C, from_cuda(out).view(np.uint32)) == want
    finally:
        torch.cuda.synchronize()
        gpu_lib.ecc_bases_destroy(h)

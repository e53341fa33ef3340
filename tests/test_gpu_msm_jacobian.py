"""The MSM's Jacobian accumulation and reduction tree at the edges of their plans: chunks
of 8 to 32 entries, one and two passes of the tree, buckets with very many or equal
partial sums.  Points are a_i G, so the sum is (sum k_i a_i) G."""
import numpy as np
import pytest

from oracle import curves, ec
from paper_2501_03245_gb300 import synth
from tests.helpers import from_cuda, limbs_to_points, to_cuda

pytestmark = pytest.mark.gpu


def _points(lib, cid, a):
    import torch

    out = torch.empty((len(a), 2 * curves.BY_ID[cid].limbs), dtype=torch.int32, device="cuda")
    lib.ecc_fixed_base_mul(cid, len(a), to_cuda(synth.ints_to_limbs(a, 8)), out)
    return out


def _check(lib, cid, a, k, pts=None):
    import torch

    C = curves.BY_ID[cid]
    pts = _points(lib, cid, a) if pts is None else pts
    out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")
    lib.ecc_msm(cid, len(a), pts, to_cuda(synth.ints_to_limbs(k, 8)), out)
    want = ec.mul(C, sum(x * y for x, y in zip(a, k)) % C.n, C.G)
    assert limbs_to_points(C, from_cuda(out).view(np.uint32))[0] == want


def _ints(q, n, seed):
    raw = np.random.default_rng(seed).bytes(40 * n)
    return [int.from_bytes(raw[40 * i:40 * i + 40], "little") % q for i in range(n)]


@pytest.mark.parametrize("cid,n", [(2, 1 << 13), (2, 140001), (2, 300007), (3, 70001), (3, 270001)])
def test_sizes(gpu_lib, cid, n):
    C = curves.BY_ID[cid]
    _check(gpu_lib, cid, _ints(C.n, n, n), _ints(C.n, n, n + 1))


@pytest.mark.parametrize("cid", [2, 3])
@pytest.mark.parametrize("c", [2, 3, 8, 9, 10, 13, 16])
def test_tree_passes(gpu_lib, cid, c):
    C = curves.BY_ID[cid]
    n = 600
    a, k = _ints(C.n, n, c), _ints(C.n, n, 50 + c)
    pts = _points(gpu_lib, cid, a)
    try:
        gpu_lib.ecc_msm_set_window(cid, 9, c)
        for chunk in (0, 1, 3, 10):
            gpu_lib.ecc_msm_set_reduce_chunk(cid, 9, chunk)
            _check(gpu_lib, cid, a, k, pts)
    finally:
        gpu_lib.ecc_msm_set_window(cid, 9, 0)
        gpu_lib.ecc_msm_set_reduce_chunk(cid, 9, 0)


@pytest.mark.parametrize("cid", [2, 3])
def test_heavy_buckets(gpu_lib, cid):
    """One scalar for all, one point for all (every addition of a bucket a doubling),
    P and -P in turn (every pair cancels), and a lone point."""
    C = curves.BY_ID[cid]
    n = 9001
    a = _ints(C.n, n, 3)
    k = _ints(C.n, 1, 4)[0]
    _check(gpu_lib, cid, a, [k] * n)
    _check(gpu_lib, cid, [a[0]] * n, [k] * n)
    _check(gpu_lib, cid, [a[0]] * n, [1] * n)
    _check(gpu_lib, cid, [a[0] if i & 1 else C.n - a[0] for i in range(n)], [k] * n)
    _check(gpu_lib, cid, a, [0] * (n - 1) + [k])
    _check(gpu_lib, cid, a, [(C.n - 1 if i & 1 else 1) for i in range(n)])


def test_split_scalars_fall_back_when_the_workspace_is_refused(gpu_lib):
    """An allocator that refuses the first request (the split form's, with the points'
    images): the call answers alike without them, from host and device offsets."""
    import torch

    C = curves.BY_ID[2]
    n = 5000
    a, k = _ints(C.n, n, 11), _ints(C.n, n, 12)
    pts, sc = _points(gpu_lib, 2, a), to_cuda(synth.ints_to_limbs(k, 8))
    want = ec.mul(C, sum(x * y for x, y in zip(a, k)) % C.n, C.G)
    offs = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    for dev in (False, True):
        sizes, held = [], {}

        def alloc(nbytes, stream):
            sizes.append(nbytes)
            if len(sizes) == 1:
                return 0
            t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
            held[t.data_ptr()] = t
            return t.data_ptr()

        def release(ptr, stream):
            torch.cuda.synchronize()
            held.pop(ptr)

        out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")
        gpu_lib.ecc_set_allocator(alloc, release)
        try:
            if dev:
                gpu_lib.ecc_msm_ragged_dev(2, 1, n, offs, pts, sc, out, 0)
            else:
                gpu_lib.ecc_msm(2, n, pts, sc, out)
            torch.cuda.synchronize()
        finally:
            gpu_lib.ecc_set_allocator(None, None)
        assert len(sizes) > 1 and not held
        assert limbs_to_points(C, from_cuda(out).view(np.uint32))[0] == want, dev

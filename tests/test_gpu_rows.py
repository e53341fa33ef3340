"""The kernels on row-major arrays (field operations, batch inversion, point addition
and doubling) where their paths divide: more elements than threads, 4-byte aligned
rows, outputs over inputs, limbs at or above the modulus, exceptional operands at the
edges of a warp and of the grid.  Exact integers are the reference."""
import numpy as np
import pytest

from oracle import curves, ec
from paper_2501_03245_gb300 import synth
from tests.helpers import from_cuda, limbs_to_points, points_to_limbs, random_points, to_cuda

pytestmark = pytest.mark.gpu
GRID = 152 * 512  # threads of a full grid


def _vals(q, n, seed):
    raw = np.random.default_rng(seed).bytes(64 * n)
    return [int.from_bytes(raw[64 * i:64 * i + 64], "little") % q for i in range(n)]


def _shift(t, words):
    """The same values in a buffer that starts `words` words past an aligned address."""
    import torch

    buf = torch.zeros(t.numel() + words, dtype=t.dtype, device="cuda")
    v = buf[words:]
    v.copy_(t.reshape(-1))
    return v.reshape(t.shape)


@pytest.mark.parametrize("cid,f", [(0, 0), (1, 0), (2, 0), (3, 0), (3, 1), (4, 1)])
@pytest.mark.parametrize("off", [0, 1])
def test_inverse_rows(gpu_lib, cid, f, off):
    import torch

    C = curves.BY_ID[cid]
    q, m = (C.p, C.limbs) if f == 0 else (C.n, 8)
    n = 1200
    X = _vals(q, n, 17 + cid)
    for i in (0, 7, 8, 31, 32, 255, 256, n - 1):
        X[i] = 0
    X[5], X[6] = q - 1, 1
    want = [pow(x, -1, q) if x else 0 for x in X]
    given = list(X)
    if q + X[9] < 1 << (32 * m):
        given[9] = q + X[9]  # not canonical
        given[0] = q         # 0 mod q
    x = _shift(to_cuda(synth.ints_to_limbs(given, m)), off)
    for fn in (gpu_lib.ecc_fp_inv, gpu_lib.ecc_fp_inv_batch, gpu_lib.ecc_fp_inv_batch_noalloc):
        out = _shift(torch.zeros_like(x), off)
        fn(cid, f, n, x, out)
        assert synth.limbs_to_ints(from_cuda(out).view(np.uint32)) == want
        same = _shift(x, off)
        fn(cid, f, n, same, same)  # in place
        assert synth.limbs_to_ints(from_cuda(same).view(np.uint32)) == want
    buf = torch.zeros((n + 3, m), dtype=x.dtype, device="cuda")
    buf[:n] = x
    gpu_lib.ecc_fp_inv_batch(cid, f, n, buf[:n], buf[3:])  # over its own input, shifted
    assert synth.limbs_to_ints(from_cuda(buf[3:].contiguous()).view(np.uint32)) == want


@pytest.mark.parametrize("n", [GRID - 1, GRID + 1, 4 * GRID + 3])
def test_inverse_past_the_grid(gpu_lib, n):
    import torch

    C = curves.BY_ID[3]
    x = to_cuda(synth.ints_to_limbs(_vals(C.n, n, n), 8))
    one = torch.zeros_like(x)
    one[:, 0] = 1
    inv, prod = torch.empty_like(x), torch.empty_like(x)
    for fn in (gpu_lib.ecc_fp_inv, gpu_lib.ecc_fp_inv_batch):
        fn(3, 1, n, x, inv)
        gpu_lib.ecc_fp_mul(3, 1, n, x, inv, prod)
        assert torch.equal(prod, one)


@pytest.mark.parametrize("cid", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("off", [0, 1])
def test_point_rows(gpu_lib, cid, off):
    import torch

    C = curves.BY_ID[cid]
    n = 600
    P, _ = random_points(C, n, 31 + cid)
    Q, _ = random_points(C, n, 77 + cid)
    for i in (0, 8, 255, n - 1):
        Q[i] = P[i]
    for i in (1, 31, 256):
        Q[i] = ec.neg(C, P[i])
    for i in (2, 32):
        P[i] = None
    for i in (3, 32, 33):
        Q[i] = None
    add, dbl = [ec.add(C, a, b) for a, b in zip(P, Q)], [ec.add(C, a, a) for a in P]
    p, q = (_shift(to_cuda(points_to_limbs(C, v)), off) for v in (P, Q))

    def check(got, want):
        assert limbs_to_points(C, from_cuda(got.contiguous()).view(np.uint32)) == want

    out = _shift(torch.zeros_like(p), off)
    gpu_lib.ecc_point_add_batch(cid, n, p, q, out)
    check(out, add)
    gpu_lib.ecc_point_dbl_batch(cid, n, p, out)
    check(out, dbl)
    same = _shift(q, off)
    gpu_lib.ecc_point_add_batch(cid, n, p, same, same)
    check(same, add)
    buf = torch.zeros((n + 2, p.shape[1]), dtype=p.dtype, device="cuda")
    buf[:n] = p
    gpu_lib.ecc_point_add_batch(cid, n, buf[:n], q, buf[2:])
    check(buf[2:], add)
    buf[:n] = q
    gpu_lib.ecc_point_add_batch(cid, n, p, buf[:n], buf[2:])
    check(buf[2:], add)


def test_point_add_past_the_grid(gpu_lib):
    """(k + 1) G = k G + G for more points than the grid has threads."""
    import torch

    n = 2 * GRID + 5
    k = np.zeros((n + 1, 8), np.uint32)
    k[:, 0] = np.arange(1, n + 2)
    pts = torch.empty((n + 1, 24), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(3, n + 1, to_cuda(k), pts)
    out = torch.empty((n, 24), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_point_add_batch(3, n, pts[:n], pts[:1].repeat(n, 1), out)
    assert torch.equal(out, pts[1:])

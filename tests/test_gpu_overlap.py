"""Results written over the inputs' own memory, whose rows have another size or start
elsewhere: k G over its scalars, signatures and keys over private keys, hashes and
nonces, verdicts over any input.  Batches of quads, of one thread an item, and past the
threads the GPU holds at once, against the same call with separate memory."""
import numpy as np
import pytest

from oracle import curves
from paper_2501_03245_gb300 import synth
from tests.helpers import to_cuda

pytestmark = pytest.mark.gpu
SIZES = [300, 9729, 160001]


def _buf(n):
    import torch

    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def _rows(C, n, seed):
    k = synth.uniform_limbs(seed, 1, n, C.n, lo=1)
    return to_cuda(np.ascontiguousarray(synth.limbs_to_be32(k)))


@pytest.mark.parametrize("cid", [1, 3])
@pytest.mark.parametrize("n", SIZES)
def test_fpmul_over_its_scalars(gpu_lib, cid, n):
    import torch

    C = curves.BY_ID[cid]
    k = to_cuda(synth.uniform_limbs(17, 1, n, C.n).view(np.uint8).reshape(n, 32))
    w = 8 * C.limbs
    want = _buf(n * w)
    gpu_lib.ecc_fixed_base_mul(cid, n, k, want)
    for off in (0, 4, 32 * n, (w - 32) * n):  # the scalars' place in the results
        buf = _buf(n * w + 64)
        src = buf[off:off + 32 * n]
        src.copy_(k.reshape(-1))
        gpu_lib.ecc_fixed_base_mul(cid, n, src, buf[:n * w])
        assert torch.equal(buf[:n * w], want), off


@pytest.mark.parametrize("cid", [0, 4])
@pytest.mark.parametrize("n", SIZES)
def test_sign_over_its_inputs(gpu_lib, cid, n):
    import torch

    C = curves.BY_ID[cid]
    ins = [_rows(C, n, 5 + i) for i in range(3)]  # d, e, k
    want = [_buf(32 * n), _buf(32 * n), _buf(64 * n)]
    gpu_lib.ecc_sign_batch(cid, n, *ins, *want)
    # offsets of d, e, k and of r, s, pub in one buffer
    for di, do in (((0, 32 * n, 64 * n), (96 * n, 128 * n, 0)), ((0, 32 * n, 64 * n), (96 * n, 128 * n, 32 * n)),
                   ((64, 32 * n + 64, 64 * n + 64), (0, 32 * n, 64 * n)), ((0, 32 * n, 64 * n), (64 * n, 0, 96 * n))):
        buf = _buf(160 * n + 128)
        src = [buf[o:o + 32 * n] for o in di]
        out = [buf[o:o + w * n] for o, w in zip(do, (32, 32, 64))]
        for a, b in zip(src, ins):
            a.copy_(b.reshape(-1))
        gpu_lib.ecc_sign_batch(cid, n, *src, *out)
        for got, ref in zip(out, want):
            assert torch.equal(got, ref), (di, do)


@pytest.mark.parametrize("cid", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_verify_over_its_inputs(gpu_lib, cid, n):
    import torch

    C = curves.BY_ID[cid]
    d, e, k = (_rows(C, n, 25 + i) for i in range(3))
    r, s, pub = _buf(32 * n), _buf(32 * n), _buf(64 * n)
    gpu_lib.ecc_sign_batch(cid, n, d, e, k, r, s, pub)
    r[::5 * 32] ^= 1
    want = _buf(n)
    gpu_lib.ecc_verify_batch(cid, n, e, r, s, pub, want)
    assert int(want.sum()) == n - (n + 4) // 5
    for at in (0, 32 * n, 64 * n, 96 * n, 31 * n, 159 * n):  # in the hashes, r, s, keys, over two of them, at the end
        buf = torch.cat([x.reshape(-1) for x in (e, r, s, pub)])
        args = [buf[a:b] for a, b in ((0, 32 * n), (32 * n, 64 * n), (64 * n, 96 * n), (96 * n, 160 * n))]
        ok = buf[at:at + n]
        gpu_lib.ecc_verify_batch(cid, n, *args, ok)
        assert torch.equal(ok, want), at

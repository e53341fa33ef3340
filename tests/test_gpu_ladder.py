"""Scalar multiplications by one thread in Jacobian coordinates: digits at the
edges of the signed windows, additions that meet equal and opposite points, and
batches around the CTA and grid sizes.  Results are exact integers, so every
comparison is exact."""
import numpy as np
import pytest

from oracle import cpp_oracle, curves, ec
from paper_2501_03245_gb300 import synth
from tests.helpers import from_cuda, to_cuda

pytestmark = pytest.mark.gpu


def edge_scalars(n):
    every = lambda h: sum(h << (16 * j) for j in range(16))  # noqa: E731
    ks = [0, 1, 2, 0x7FFF, 0x8000, 0x8001, 0xFFFF, 0x10000, n - 1, n - 2, n - 0x8000, n, n + 1, n // 2,
          n // 2 + 1, 1 << 255, (1 << 256) - 1]
    ks += [every(h) for h in (0x7FFF, 0x8000, 0x8001, 0xFFFF)] + [every(0x8000) >> 1, n - every(0x7FFF) % n]
    ks += [0x8000 << (16 * j) for j in range(16)] + [n - (1 << (16 * j)) for j in range(16)]
    return ks


@pytest.mark.parametrize("cid", [0, 1, 2, 3, 4])
def test_fpmul_edge_digits(gpu_lib, cid):
    import torch

    C = curves.BY_ID[cid]
    ks = edge_scalars(C.n)
    out = torch.zeros((len(ks), 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(cid, len(ks), to_cuda(synth.ints_to_limbs(ks, 8)), out)
    torch.cuda.synchronize()
    want = [ec.encode(ec.mul(C, k % C.n, C.G)) for k in ks]
    got = from_cuda(out).view(np.uint32)
    assert synth.limbs_to_ints(got[:, :C.limbs]) == [w[0] for w in want]
    assert synth.limbs_to_ints(got[:, C.limbs:]) == [w[1] for w in want]


def triples(cid, dus):
    """A valid triple for every (d, u1, u2): r = x(u1 G + u2 Q), s = r / u2, e = u1 s
    (r = 1 where the sum is O, which is to be refused)."""
    C = curves.BY_ID[cid]
    rows = []
    for d, u1, u2 in dus:
        R = ec.mul(C, (u1 + u2 * d) % C.n, C.G)
        r = R[0] % C.n if R else 1
        s = r * pow(u2, -1, C.n) % C.n
        rows.append((u1 * s % C.n, r, s, ec.mul(C, d, C.G)))
    be = lambda v: synth.limbs_to_be32(synth.ints_to_limbs(v, 8))  # noqa: E731
    e, r, s = (be([row[i] for row in rows]) for i in range(3))
    pub = np.concatenate([be([row[3][0] for row in rows]), be([row[3][1] for row in rows])], axis=1)
    return e, r, s, pub


@pytest.mark.parametrize("cid", [0, 1, 4])
def test_verify_edge_digits_and_colliding_points(gpu_lib, cid):
    """u1 G and u2 Q equal, opposite, zero or table points; windows of every value."""
    import torch

    n = curves.BY_ID[cid].n
    w5 = lambda d: sum(d << (5 * i) for i in range(51)) % n  # noqa: E731
    us = [1, 2, 15, 16, 17, 31, 32, n - 1, n - 16, n - 17, n // 2, 1 << 254, w5(15), w5(16), w5(17), w5(31)]
    dus = [(d, u1, u2) for d in (1, n - 1, 2, 16, 0x8000, n // 2) for u2 in us
           for u1 in (0, 1, 0x8000, u2 * d % n, -u2 * d % n)]
    e, r, s, pub = triples(cid, dus)
    bad = r.copy()
    bad[:, 31] ^= 1
    e, r, s, pub = (np.concatenate(p) for p in ((e, e), (r, bad), (s, s), (pub, pub)))
    ok = torch.zeros(len(e), dtype=torch.uint8, device="cuda")
    gpu_lib.ecc_verify_batch(cid, len(e), to_cuda(e), to_cuda(r), to_cuda(s), to_cuda(pub), ok)
    torch.cuda.synchronize()
    want = cpp_oracle.verify(cid, e, r, s, pub)
    assert np.array_equal(from_cuda(ok), want)
    assert want[: len(dus)].sum() >= 3 * len(dus) // 4 and want[len(dus):].sum() == 0


@pytest.mark.parametrize("n", [127, 128, 129, 152 * 512 + 1])
def test_verify_sizes(gpu_lib, n):
    """A CTA's and a full grid's edges: rows repeat 40 triples, every third one damaged."""
    import torch

    e, r, s, pub = triples(1, [(3 + 7 * i, 5 + i * i, 11 + 3 * i) for i in range(40)])
    s[::3, 5] ^= 4
    idx = np.arange(n) * 13 % 40
    ok = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    gpu_lib.ecc_verify_batch(1, n, *(to_cuda(np.ascontiguousarray(a[idx])) for a in (e, r, s, pub)), ok)
    torch.cuda.synchronize()
    assert np.array_equal(from_cuda(ok), (idx % 3 != 0).astype(np.uint8))


@pytest.mark.parametrize("cid", [0, 1, 4])
def test_quads_and_threads_agree(gpu_lib, cid):
    """The largest batches that eight and four lanes verify an item of, and one more, with
    the edge digits and colliding points in the rows of all."""
    import torch

    n = curves.BY_ID[cid].n
    us = [1, 16, 17, n - 1, n - 17, n // 2]
    dus = [(d, u1, u2) for d in (1, n - 1, 16) for u2 in us for u1 in (0, 1, 0x8000, u2 * d % n, -u2 * d % n)]
    e, r, s, pub = triples(cid, dus)
    r[1::7, 31] ^= 1
    want = cpp_oracle.verify(cid, e, r, s, pub)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for m in (1, 15, 17, 33, 16 * sms, 16 * sms + 1, 64 * sms, 64 * sms + 1):
        idx = np.arange(m) * 11 % len(e)
        ok = torch.full((m,), 7, dtype=torch.uint8, device="cuda")
        gpu_lib.ecc_verify_batch(cid, m, *(to_cuda(np.ascontiguousarray(a[idx])) for a in (e, r, s, pub)), ok)
        torch.cuda.synchronize()
        assert np.array_equal(from_cuda(ok), want[idx]), m


@pytest.mark.parametrize("cid", [0, 1, 2, 3, 4])
def test_fpmul_and_sign_by_quads_and_threads(gpu_lib, cid):
    """k G at the largest batch of quads, one more and the first sizes of a CTA, with the
    edge digits in every batch; signatures with the same nonces, their r is x(k G)."""
    import torch

    C = curves.BY_ID[cid]
    ks = [k for k in edge_scalars(C.n) if 0 < k < C.n]
    want = [ec.encode(ec.mul(C, k, C.G)) for k in ks]
    wx, wy = (np.array([synth.ints_to_limbs([w[i]], C.limbs)[0] for w in want]) for i in (0, 1))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for m in (1, 31, 33, 64 * sms, 64 * sms + 1):
        idx = np.arange(m) * 7 % len(ks)
        limbs = synth.ints_to_limbs(ks, 8)[idx]
        out = torch.zeros((m, 2 * C.limbs), dtype=torch.int32, device="cuda")
        gpu_lib.ecc_fixed_base_mul(cid, m, to_cuda(limbs), out)
        got = from_cuda(out).view(np.uint32)
        assert np.array_equal(got[:, :C.limbs], wx[idx]) and np.array_equal(got[:, C.limbs:], wy[idx]), m
        if cid not in (0, 1, 4):
            continue
        k = to_cuda(np.ascontiguousarray(synth.limbs_to_be32(limbs)))
        e = k.flip(0).contiguous()
        d = k.clone()
        r, pub = torch.zeros_like(k), torch.zeros((m, 64), dtype=torch.uint8, device="cuda")
        s = d  # over the private keys' own buffer
        gpu_lib.ecc_sign_batch(cid, m, d, e, k, r, s, pub)
        assert np.array_equal(from_cuda(pub)[:, :32], synth.limbs_to_be32(wx[idx]))
        rows = range(min(m, len(ks)))
        for i in rows:
            kk, h = ks[idx[i]], ks[idx[m - 1 - i]]
            rr = want[idx[i]][0] % C.n
            assert int.from_bytes(bytes(from_cuda(r[i])), "big") == rr
            assert int.from_bytes(bytes(from_cuda(s[i])), "big") == pow(kk, -1, C.n) * (h + rr * kk) % C.n

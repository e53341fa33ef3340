"""Calls whose workspace is bounded (an allocator that refuses what passes its budget).
The budgets are what the calls took when their plans knew one form only: faster forms
that want more are given up where they are refused, and the results stay."""
import numpy as np
import pytest

from oracle import curves, ec
from paper_2501_03245_gb300 import synth
from tests.helpers import from_cuda, limbs_to_points, to_cuda

pytestmark = pytest.mark.gpu


class Arena:
    """A workspace allocator of `budget` bytes in all."""

    def __init__(self, lib, budget):
        self.lib, self.budget, self.used, self.held, self.refused = lib, budget, 0, {}, 0

    def __enter__(self):
        self.lib.ecc_set_allocator(self.alloc, self.release)
        return self

    def __exit__(self, *exc):
        self.lib.ecc_set_allocator(None, None)
        return False

    def alloc(self, nbytes, stream):
        import torch

        if self.used + nbytes > self.budget:
            self.refused += 1
            return 0
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        self.used += nbytes
        self.held[t.data_ptr()] = t
        return t.data_ptr()

    def release(self, ptr, stream):
        import torch

        torch.cuda.synchronize()
        self.used -= self.held.pop(ptr).numel()


def _points(lib, cid, n):
    import torch

    a = np.zeros((n, 8), np.uint32)
    a[:, 0] = np.arange(1, n + 1)
    out = torch.empty((n, 2 * curves.BY_ID[cid].limbs), dtype=torch.int32, device="cuda")
    lib.ecc_fixed_base_mul(cid, n, to_cuda(a), out)
    return out


def _scalars(C, n, seed):
    k = synth.uniform_limbs(seed, 1, n, C.n)
    return to_cuda(k.view(np.int32)), synth.limbs_to_ints(k)


def _check(C, out, totals):
    got = limbs_to_points(C, from_cuda(out).view(np.uint32))
    assert got == [ec.mul(C, t % C.n, C.G) if t % C.n else None for t in totals]


@pytest.mark.parametrize("cid,n,budget", [(2, 1, 89472), (2, 4096, 2476800), (2, 1 << 15, 15504128),
                                          (2, 1 << 18, 99645184), (3, 1, 125504), (3, 256, 428368),
                                          (3, 4096, 3369856), (3, 1 << 15, 21169920)])
def test_msm(gpu_lib, cid, n, budget):
    import torch

    C = curves.BY_ID[cid]
    pts = _points(gpu_lib, cid, n)
    kd, k = _scalars(C, n, 7)
    total = sum((i + 1) * x for i, x in enumerate(k))
    out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")
    with Arena(gpu_lib, budget) as arena:
        gpu_lib.ecc_msm(cid, n, pts, kd, out)
        torch.cuda.synchronize()
    assert arena.refused and not arena.held
    _check(C, out, [total])


@pytest.mark.parametrize("cid,n,c,vectors,budget", [(2, 4096, 0, 4, 8846336), (3, 4096, 0, 4, 11893760),
                                                    (2, 4096, 16, 1, 5050624), (3, 1 << 16, 16, 1, 20058368)])
def test_bases(gpu_lib, cid, n, c, vectors, budget):
    import torch

    C = curves.BY_ID[cid]
    kd, k = _scalars(C, n * vectors, 8)
    totals = [sum((i + 1) * x for i, x in enumerate(k[v * n:(v + 1) * n])) for v in range(vectors)]
    out = torch.zeros((vectors, 2 * C.limbs), dtype=torch.int32, device="cuda")
    h = gpu_lib.ecc_bases_create(cid, n, _points(gpu_lib, cid, n))
    try:
        if c:
            gpu_lib.ecc_bases_precompute(h, c)
        with Arena(gpu_lib, budget) as arena:
            gpu_lib.ecc_msm_bases(h, vectors, kd, out)
            torch.cuda.synchronize()
            assert arena.refused
            _check(C, out, totals)
            sizes = torch.full((vectors,), n, dtype=torch.int64, device="cuda")
            gpu_lib.ecc_msm_bases_ragged_dev(h, vectors, n * vectors, sizes, kd, out.zero_())
            torch.cuda.synchronize()
        assert not arena.held
    finally:
        gpu_lib.ecc_bases_destroy(h)
    _check(C, out, totals)


@pytest.mark.parametrize("cid,num,per,budget", [(2, 1024, 64, 158256384), (3, 300, 1, 36558592)])
def test_ragged(gpu_lib, cid, num, per, budget):
    """A budget that may or may not be passed: host and device offsets answer alike."""
    import torch

    C = curves.BY_ID[cid]
    n = num * per
    pts = _points(gpu_lib, cid, n)
    kd, k = _scalars(C, n, 9)
    totals = [sum((i + 1) * k[i] for i in range(v * per, (v + 1) * per)) for v in range(num)]
    offs = np.arange(num + 1, dtype=np.uint64) * per
    out = torch.zeros((num, 2 * C.limbs), dtype=torch.int32, device="cuda")
    with Arena(gpu_lib, budget) as arena:
        gpu_lib.ecc_msm_ragged(cid, num, offs, pts, kd, out)
        torch.cuda.synchronize()
        _check(C, out, totals)
        gpu_lib.ecc_msm_ragged_dev(cid, num, n, to_cuda(offs.view(np.int64)), pts, kd, out.zero_(), 0)
        torch.cuda.synchronize()
    assert not arena.held
    _check(C, out, totals)


@pytest.mark.parametrize("cid", [0, 1])
@pytest.mark.parametrize("n,budget", [(33, 45301), (1000, 1365256), (9728, 13278976), (30000, 40950256),
                                      (77825, 106231381), (9728, 100000), (77825, 2000000)])
def test_verify(gpu_lib, cid, n, budget):
    """Fewer items at once, by eight, four and one lanes: as with the full workspace."""
    import torch

    C = curves.BY_ID[cid]
    d, e, k = (to_cuda(np.ascontiguousarray(synth.limbs_to_be32(synth.uniform_limbs(3 + i, 1, n, C.n, lo=1))))
               for i in range(3))
    r, s = torch.empty_like(d), torch.empty_like(d)
    pub = torch.empty((n, 64), dtype=torch.uint8, device="cuda")
    gpu_lib.ecc_sign_batch(cid, n, d, e, k, r, s, pub)
    s[::7, 3] ^= 16
    ok = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    with Arena(gpu_lib, budget) as arena:
        gpu_lib.ecc_verify_batch(cid, n, e, r, s, pub, ok)
        torch.cuda.synchronize()
    assert arena.refused and not arena.held
    assert np.array_equal(from_cuda(ok), (np.arange(n) % 7 != 0).astype(np.uint8))


@pytest.mark.parametrize("cid", [2, 3])
def test_graph_recorded_before_a_window_table(gpu_lib, cid):
    """A call recorded on a handle replays on new scalars after the handle got a window
    table: what it reads stays where it was."""
    import torch

    C, n = curves.BY_ID[cid], 3000
    ks = [_scalars(C, n, s) for s in (20, 21)]
    out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")
    h = gpu_lib.ecc_bases_create(cid, n, _points(gpu_lib, cid, n))
    try:
        kd = ks[0][0].clone()
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            gpu_lib.ecc_msm_bases(h, 1, kd, out, s)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            gpu_lib.ecc_msm_bases(h, 1, kd, out, s)
        gpu_lib.ecc_bases_precompute(h, 12)
        kd.copy_(ks[1][0])
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        _check(C, out, [sum((i + 1) * x for i, x in enumerate(ks[1][1]))])
        gpu_lib.ecc_msm_bases(h, 1, ks[0][0], out.zero_())
        _check(C, out, [sum((i + 1) * x for i, x in enumerate(ks[0][1]))])
        del g
    finally:
        torch.cuda.synchronize()
        gpu_lib.ecc_bases_destroy(h)

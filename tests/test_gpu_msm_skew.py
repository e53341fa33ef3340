"""MSMs whose entries fall into few buckets (scalars of zeros and ones, a nearly empty top
window): the closed form, and no CTA of the fold is left to walk the empty buckets."""
import numpy as np
import pytest

from oracle import curves, ec
from paper_2501_03245_gb300 import synth
from tests.helpers import from_cuda, limbs_to_points, to_cuda

pytestmark = pytest.mark.gpu


def _multiples(n):
    a = np.zeros((n, 8), np.uint32)
    a[:, 0] = np.arange(1, n + 1)
    return a


def _fold_ms(lib, call):
    best = None
    for _ in range(4):
        call()
        t = lib.ecc_msm_phase_times()["fold"]
        best = t if best is None else min(best, t)
    return best


@pytest.mark.parametrize("cid", [2, 3])
def test_zeros_and_ones_on_a_window_table(gpu_lib, cid):
    """4 vectors cost no more than 4 times one, and a millisecond; by slots alone the empty
    buckets between the vectors' first ones went to one CTA each (8 ms against 0.1)."""
    import torch

    C, n, V = curves.BY_ID[cid], 4096, 4
    a = _multiples(n)
    pts = torch.empty((n, 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(cid, n, to_cuda(a), pts)
    k = np.zeros((V * n, 8), np.uint32)
    k[:, 0] = np.random.default_rng(cid).integers(0, 2, V * n)
    kd = to_cuda(k)
    out = torch.zeros((V, 2 * C.limbs), dtype=torch.int32, device="cuda")
    h = gpu_lib.ecc_bases_create(cid, n, pts)
    try:
        gpu_lib.ecc_bases_precompute(h, 20)
        gpu_lib.ecc_set_phase_timing(1)
        one = _fold_ms(gpu_lib, lambda: gpu_lib.ecc_msm_bases(h, 1, kd[:n], out[:1]))
        four = _fold_ms(gpu_lib, lambda: gpu_lib.ecc_msm_bases(h, V, kd, out))
    finally:
        gpu_lib.ecc_set_phase_timing(0)
        torch.cuda.synchronize()
        gpu_lib.ecc_bases_destroy(h)
    got = limbs_to_points(C, from_cuda(out).view(np.uint32))
    for v in range(V):
        total = int((a[:, 0].astype(np.int64) * k[v * n:(v + 1) * n, 0]).sum())
        assert got[v] == ec.mul(C, total % C.n, C.G), v
    assert four < 4 * one + 1.0, (one, four)


@pytest.mark.parametrize("cid", [2, 3])
def test_nearly_empty_top_window(gpu_lib, cid):
    """Uniform scalars and 20-bit windows: few values of the top window hold a row's
    entries, the rest of its buckets are empty."""
    import torch

    C, n = curves.BY_ID[cid], 1 << 16
    a = _multiples(n)
    pts = torch.empty((n, 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(cid, n, to_cuda(a), pts)
    k = synth.uniform_limbs(91, 1, n, C.n)
    kd = to_cuda(k.view(np.int32))
    out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_msm_set_window(cid, 16, 20)
    try:
        gpu_lib.ecc_set_phase_timing(1)
        t = _fold_ms(gpu_lib, lambda: gpu_lib.ecc_msm(cid, n, pts, kd, out))
    finally:
        gpu_lib.ecc_set_phase_timing(0)
        gpu_lib.ecc_msm_set_window(cid, 16, 0)
    total = sum(int(x) * y for x, y in zip(a[:, 0], synth.limbs_to_ints(k)))
    assert limbs_to_points(C, from_cuda(out).view(np.uint32))[0] == ec.mul(C, total % C.n, C.G)
    assert t < 2.0, t  # 8.1 (BN254) and 3.0 ms (BLS12-381) by slots alone, 0.5 and 0.8 now


def test_batches_of_tiny_msms(gpu_lib):
    """16384 BLS12-381 MSMs of 0 to 4 points: every one right, and no slower than with the
    4-bit windows that are too wide for them (16 buckets a row for 4 entries)."""
    import torch

    cid, C, num = 3, curves.BLS12_381, 16384
    sizes = np.arange(num) % 5
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    n = int(offs[-1])
    pts = torch.empty((n, 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(cid, n, to_cuda(_multiples(n)), pts)
    k = synth.uniform_limbs(92, 1, n, C.n)
    kd, ks = to_cuda(k.view(np.int32)), synth.limbs_to_ints(k)
    totals = [sum((i + 1) * ks[i] for i in range(int(a), int(b))) % C.n for a, b in zip(offs[:-1], offs[1:])]
    want = torch.empty((num, 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(cid, num, to_cuda(synth.ints_to_limbs(totals, 8).view(np.int32)), want)

    def run():
        out = torch.zeros_like(want)
        ms = []
        for _ in range(4):
            gpu_lib.ecc_msm_ragged(cid, num, offs, pts, kd, out)
            ms.append(sum(gpu_lib.ecc_msm_phase_times().values()))
        assert torch.equal(out, want)
        return min(ms)

    try:
        gpu_lib.ecc_set_phase_timing(1)
        own = run()
        for lg in (1, 2):
            gpu_lib.ecc_msm_set_window(cid, lg, 4)
        wide = run()
    finally:
        gpu_lib.ecc_set_phase_timing(0)
        for lg in (1, 2):
            gpu_lib.ecc_msm_set_window(cid, lg, 0)
    assert own < 0.9 * wide, (own, wide)


def test_split_or_whole_scalars(gpu_lib):
    """BN254 on each side of the size up to which scalars are split, and with 18-bit windows,
    whose halves' top window holds only a carry: right either way, and no slower at 18
    bits than the halves were (19 ms for 2^22 points against 12 with 19 bits)."""
    import torch

    cid, C, n_max = 2, curves.BN254, 1 << 22
    a = _multiples(n_max)
    pts = torch.empty((n_max, 2 * C.limbs), dtype=torch.int32, device="cuda")
    gpu_lib.ecc_fixed_base_mul(cid, n_max, to_cuda(a), pts)
    k = synth.uniform_limbs(93, 1, n_max, C.n)
    kd = to_cuda(k.view(np.int32))
    out = torch.zeros((1, 2 * C.limbs), dtype=torch.int32, device="cuda")

    def run(n, c):
        gpu_lib.ecc_msm_set_window(cid, n.bit_length() - 1, c)
        ms = []
        for _ in range(4):
            gpu_lib.ecc_msm(cid, n, pts[:n], kd[:n], out)
            ms.append(sum(gpu_lib.ecc_msm_phase_times().values()))
        gpu_lib.ecc_msm_set_window(cid, n.bit_length() - 1, 0)
        total = 0
        for j in range(8):  # 16-bit halves of the limbs: every partial sum fits 64 bits
            for h in (0, 16):
                v = (k[:n, j] >> h & 0xFFFF).astype(np.int64)
                total += int((v * a[:n, 0].astype(np.int64)).sum()) << (32 * j + h)
        assert limbs_to_points(C, from_cuda(out).view(np.uint32))[0] == ec.mul(C, total % C.n, C.G), (n, c)
        return min(ms)

    try:
        gpu_lib.ecc_set_phase_timing(1)
        for n, c in ((1 << 21, 0), ((1 << 21) + 1, 0), (1 << 18, 18), (1 << 18, 16), (n_max, 0)):
            run(n, c)
        t18, t19 = run(n_max, 18), run(n_max, 19)
    finally:
        gpu_lib.ecc_set_phase_timing(0)
    assert t18 < 1.35 * t19, (t18, t19)

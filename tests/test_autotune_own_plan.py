"""The tuners leave the library's own plan where no forced setting beats it, against a
fake library and clock: width 0 and chunk 0 stand for "no override"."""
import json
import types

import pytest

from paper_2501_03245_gb300 import autotune


class FakeLib:
    """Reported (textbook) widths and the overrides; a call costs cost(overrides)."""

    ECC_BN254, ECC_BLS12_381 = 2, 3

    def __init__(self, textbook):
        self.textbook, self.w, self.chunk = dict(textbook), {}, {}

    def ecc_msm_window(self, curve, n):
        l = n.bit_length() - 1
        return self.w.get(l) or self.textbook[l]

    def ecc_msm_set_window(self, curve, l, c):
        assert c == 0 or 2 <= c <= 20
        self.w[l] = c

    def ecc_msm_set_reduce_chunk(self, curve, l, k):
        assert 0 <= k <= 10
        self.chunk[l] = k

    def own_plan(self, curve, log2_sizes):
        for l in log2_sizes:
            self.w[l] = self.chunk[l] = 0

    def forced(self):
        return any(self.w.values()) or any(self.chunk.values())


def fake_torch(clock):
    class Event:
        def __init__(self, enable_timing=True):
            self.t = None

        def record(self):
            self.t = clock[0]

        def elapsed_time(self, other):
            return other.t - self.t

    class Tensor:
        cuda = contiguous = lambda self: self
        __getitem__ = lambda self, i: self

    cuda = types.SimpleNamespace(Event=Event, synchronize=lambda: None, get_device_name=lambda: "fake")
    return types.SimpleNamespace(cuda=cuda, from_numpy=lambda a: Tensor())


def batch(monkeypatch, lib, cost):
    monkeypatch.setattr(autotune, "ecc", lib)
    monkeypatch.setattr(autotune, "msm_own_plan", lib.own_plan)
    clock = [0.0]

    def run():
        clock[0] += cost(lib)

    return autotune.tune_batch(0, sorted(lib.textbook), run, fake_torch(clock))


def test_batch_keeps_the_own_plan(monkeypatch):
    """Every forced setting costs 7% more: all overrides are removed, those that were
    installed before too."""
    lib = FakeLib({10: 8, 14: 11})
    lib.ecc_msm_set_window(0, 10, 8)
    out = batch(monkeypatch, lib, lambda lib: 40.4 if lib.forced() else 37.6)
    assert out["own"] and out["shift"] is None and out["chunk_log2"] is None
    assert not lib.forced() and out["widths"] == {10: 8, 14: 11}


def test_batch_installs_what_beats_the_own_plan(monkeypatch):
    lib = FakeLib({10: 8, 14: 11})
    out = batch(monkeypatch, lib, lambda lib: 30.0 if lib.w.get(14) == 12 else 37.6)
    assert not out["own"] and out["shift"] == 1 and lib.w == {10: 9, 14: 12}


@pytest.mark.parametrize("gain,want", [(0.0, 0), (0.003, 0), (0.02, 9)])
def test_class_keeps_the_own_plan_unless_beaten(monkeypatch, tmp_path, gain, want):
    lib = FakeLib({12: 8})
    monkeypatch.setattr(autotune, "ecc", lib)
    monkeypatch.setattr(autotune, "make_bases", lambda *a: None)
    monkeypatch.setattr(autotune, "time_msm", lambda *a: {0: 1.0, 9: 1.0 - gain}.get(lib.w.get(12, 0), 1.1))
    cache = tmp_path / "t.json"
    # a table measured on former kernels is not taken over
    cache.write_text(json.dumps({"fake|2|1": {"12": 7}}))
    torch = fake_torch([0.0])
    assert autotune.tune(2, [12], torch, cache=str(cache)) == {12: want}
    assert lib.w[12] == want
    monkeypatch.setattr(autotune, "time_msm", None)  # the table is read, not measured again
    lib.w[12] = 5
    assert autotune.tune(2, [12], torch, cache=str(cache)) == {12: want} and lib.w[12] == want

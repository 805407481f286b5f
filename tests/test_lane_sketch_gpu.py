"""The lane-wide sketch (one window per lane) against the oracle where it can
go wrong: window counts around the 32 of a warp's round, rounds that cross
targets, targets too short for a window spread between others, invalid
bases, repeated k-mers, more candidates than a lane sorts, every start
alignment, and the largest windows.  Integer work: equality."""
import random

import numpy as np
import pytest

import oracle
from gpu_helpers import dev, gpu_sketch, offsets, u8

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


PARAMS = [
    dict(k=16, sketch_size=16, window_len=128, window_stride=113),
    dict(k=16, sketch_size=16, window_len=127, window_stride=112),
    dict(k=16, sketch_size=1, window_len=16, window_stride=1),
    dict(k=16, sketch_size=16, window_len=512, window_stride=497),
    dict(k=15, sketch_size=15, window_len=257, window_stride=243),
    dict(k=5, sketch_size=16, window_len=60, window_stride=7),
    dict(k=12, sketch_size=8, window_len=64, window_stride=40),
    dict(k=1, sketch_size=16, window_len=130, window_stride=130),
]


def _targets(rng, p):
    """Sequences whose windows fill, just miss and just pass whole rounds of
    32, with empty and too short ones between them."""
    k, w, st = p["k"], p["window_len"], p["window_stride"]

    def rand(n, n_rate=0.0):
        return "".join(rng.choice("N") if rng.random() < n_rate else rng.choice("ACGTacgt") for _ in range(n))

    def of_windows(n):  # a sequence of exactly n windows
        return rand((n - 1) * st + k + rng.randrange(st))

    out = [of_windows(n) for n in (1, 31, 32, 33, 63, 65)]
    for _ in range(40):  # one-window targets in a row, and gaps of targets without windows
        out += [rand(k + rng.randrange(st)), "", rand(k - 1)]
    out += [rand(k - 1) for _ in range(300)] + [of_windows(3)]
    out += [rand(40 * st, 0.002), rand(40 * st, 0.2), "N" * (5 * st), rand(20 * st, 0.01)]
    out += ["A" * (3 * w), "ACGT" * w, (rand(37) * (4 * w // 37 + 1)), "AC" * 40 + rand(w) + "T" * w]
    return out


@pytest.mark.parametrize("p", PARAMS, ids=lambda p: f"k{p['k']}s{p['sketch_size']}w{p['window_len']}st{p['window_stride']}")
def test_sketch_equals_oracle(mc, p):
    rng = random.Random(p["k"] * 1000 + p["window_len"])
    seqs = _targets(rng, p)
    seq, offs = "".join(seqs), offsets([len(s) for s in seqs])
    win, sk, cnt = gpu_sketch(mc, seq, offs, **p)
    owin, osk, ocnt = oracle.sketch(seq, offs, **p)
    assert (win == owin).all()
    assert (cnt == ocnt).all()
    assert (sk == osk).all()


@pytest.mark.parametrize("shift", [0, 1, 7, 15])
def test_build_from_any_alignment(mc, shift):
    """The bases may start at any address; the dump equals the oracle's."""
    import torch
    p = dict(PARAMS[0], bucket_cap=5)
    rng = random.Random(shift)
    seqs = _targets(rng, p)
    seq, offs = u8("".join(seqs)), offsets([len(s) for s in seqs])
    buf = torch.zeros(len(seq) + 64, dtype=torch.uint8, device="cuda")
    buf[16 + shift:16 + shift + len(seq)] = dev(seq)
    db = mc.Database.create(np.zeros(1, np.uint32), **p)
    try:
        db.add_targets(buf[16 + shift:], dev(offs), np.zeros(len(seqs), np.uint32))
        db.finalize()
        got, want = db.dump(), oracle.DB(seq, offs, **p).dump()
        for a, b in zip(got, want):
            assert len(a) == len(b) and (a == b).all()
    finally:
        db.free()


def test_overlapping_sequences_are_sketched_on_their_own(mc):
    """mc_sketch takes sequences that overlap in memory (offsets that go
    back leave an empty sequence between them)."""
    p = PARAMS[0]
    rng = random.Random(5)
    seq = "".join(rng.choice("ACGT") for _ in range(9000))
    offs = np.array([0, 4000, 300, 6000, 5990, 9000], dtype=np.uint64)
    win, sk, cnt = gpu_sketch(mc, seq, offs, **p)
    at = 0
    for a, b in zip(offs[:-1], offs[1:]):
        if b <= a:
            continue
        _, osk, ocnt = oracle.sketch(seq[int(a):int(b)], offsets([int(b - a)]), **p)
        n = len(ocnt)
        assert (cnt[at:at + n] == ocnt).all() and (sk[at:at + n] == osk).all()
        at += n
    assert at == len(cnt)

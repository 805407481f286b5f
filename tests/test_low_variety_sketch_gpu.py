"""Sketches of sequence without variety, where most windows of a warp need
the exact selection: invalid bases, short periods, few possible k-mers, and
as many such windows in a warp's round as the line between its two forms
needs.  Equal to the oracle."""
import random

import numpy as np
import pytest

import oracle
from gpu_helpers import dev, gpu_sketch, offsets, u8

pytestmark = pytest.mark.gpu
ONES = "TCCCTTGCTGTTTACA"  # the 16-mer whose hash is 0xFFFFFFFF


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


def _rand(rng, n, alphabet="ACGT"):
    return "".join(rng.choice(alphabet) for _ in range(n))


def _sequences(rng, p):
    k, w, st = p["k"], p["window_len"], p["window_stride"]
    n = 70 * st + w
    out = ["N" * n, "A" * n, "acgt" * (n // 4), "N" * (k - 1) + ONES + "N" * n, (ONES + "N") * (n // 17)]
    out += [(_rand(rng, period) * (n // period + 1))[:n] for period in (2, 3, 5, 6, 9, 15, 16, 17, 23, 40)]
    out += [_rand(rng, n, "AC"), _rand(rng, n, "AAAAAAAC"), _rand(rng, n, "ACGTN")]
    for few in range(9, 18):  # so many windows of a round of 32 without variety
        x = list(_rand(rng, 32 * st + w))
        for j in rng.sample(range(32), few):
            x[j * st: j * st + w] = (_rand(rng, 4) * (w // 4 + 1))[:w]
        out.append("".join(x))
    return out


@pytest.mark.parametrize("p", [dict(k=16, sketch_size=16, window_len=128, window_stride=113),
                               dict(k=16, sketch_size=5, window_len=40, window_stride=11),
                               dict(k=16, sketch_size=16, window_len=512, window_stride=497),
                               dict(k=15, sketch_size=15, window_len=257, window_stride=243),
                               dict(k=4, sketch_size=16, window_len=128, window_stride=125),
                               dict(k=6, sketch_size=16, window_len=128, window_stride=60),
                               dict(k=7, sketch_size=16, window_len=128, window_stride=60),
                               dict(k=9, sketch_size=16, window_len=100, window_stride=92),
                               dict(k=12, sketch_size=8, window_len=64, window_stride=40),
                               dict(k=2, sketch_size=1, window_len=50, window_stride=49),
                               dict(k=1, sketch_size=16, window_len=300, window_stride=300)],
                         ids=lambda p: f"k{p['k']}s{p['sketch_size']}w{p['window_len']}")
def test_low_variety(mc, p):
    rng = random.Random(p["k"] + p["window_len"])
    seqs = _sequences(rng, p)
    seq, offs = "".join(seqs), offsets([len(s) for s in seqs])
    win, sk, cnt = gpu_sketch(mc, seq, offs, **p)
    owin, osk, ocnt = oracle.sketch(seq, offs, **p)
    assert (win == owin).all() and (cnt == ocnt).all() and (sk == osk).all()
    # the build's form of the same kernel
    prm = dict(p, bucket_cap=5)
    db = mc.Database.create(np.zeros(1, np.uint32), **prm)
    try:
        db.add_targets(dev(u8(seq)), dev(offs), np.zeros(len(seqs), np.uint32))
        db.finalize()
        for a, b in zip(db.dump(), oracle.DB(seq, offs, **prm).dump()):
            assert len(a) == len(b) and (a == b).all()
    finally:
        db.free()


def test_hash_of_all_ones_is_a_feature(mc):
    p = dict(k=16, sketch_size=16, window_len=128, window_stride=113)
    seq = (ONES + "N") * 600
    _, sk, cnt = gpu_sketch(mc, seq, offsets([len(seq)]), **p)
    assert (cnt == 1).all() and (sk[:, 0] == 0xFFFFFFFF).all()

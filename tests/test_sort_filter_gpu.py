"""Classification's filter (locations whose target and window block are hit
too rarely to matter are dropped before the sort) against the oracle: where
the bound that guides it is tight and where it is not (tandem copies next to
each other double it), with every survivor count from none to all, location
counts around the size classes' edges, reads without a clear winner, full
candidate lists, wide sliding windows, and 64-bit locations.  Integer work:
equality."""
import random

import numpy as np
import pytest

import oracle
from gpu_helpers import dev, gpu_build, host_u32, offsets, u8

pytestmark = pytest.mark.gpu
P = dict(k=16, sketch_size=16, window_len=128, window_stride=113, bucket_cap=254)


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


def _rand(rng, n):
    return "".join(rng.choice("ACGT") for _ in range(n))


def _mutated(rng, s, rate):
    return "".join(rng.choice("ACGT") if rng.random() < rate else c for c in s)


def _targets(rng):
    root = _rand(rng, 6000)
    out = [_mutated(rng, root, r) for r in (0, 0, 0.001, 0.005, 0.01, 0.02, 0.03, 0.05, 0.08)]
    for period in (1, 2, 3, 4, 5, 8, 9):  # tandem copies at window distances around a block's size
        out.append(_rand(rng, 113 * period) * (40 // period + 2))
    unit = _rand(rng, 900)  # many copies, some of them shifted against the window grid
    out += [_rand(rng, rng.choice([0, 113, 5])) + _mutated(rng, unit, 0.002) + _rand(rng, 300) for _ in range(70)]
    out += [_rand(rng, 2000) for _ in range(10)]
    return out, unit


def _queries(rng, targets, unit):
    qs = []
    for _ in range(400):
        t = rng.choice(targets)
        n = rng.choice([40, 100, 129, 150, 250])
        a = rng.randrange(max(1, len(t) - n))
        m1 = _mutated(rng, t[a:a + n], rng.choice([0, 0.01, 0.1]))
        if rng.random() < 0.5:
            qs.append([m1])
        else:
            b = min(max(0, len(t) - n), a + rng.randrange(200))
            qs.append([m1, _mutated(rng, t[b:b + n], 0.01)])
    for _ in range(150):  # 16 to 64 features that hit up to 70 targets each
        a = rng.randrange(0, 700)
        qs.append([unit[a:a + rng.choice([60, 128, 200])], unit[rng.randrange(600):][:rng.choice([30, 128, 250])]])
    qs += [[_rand(rng, 150), _rand(rng, 150)] for _ in range(60)]
    qs += [[targets[rng.randrange(9)][50:150], _rand(rng, 100), targets[20][300:400]] for _ in range(30)]
    # invalid bases, lower case, empty and short mates, long reads, repeats, no mates
    qs += [[x[:n] + "N" + x[n + 1:].lower() for x in q] for n, q in zip(range(40), qs)]
    qs += [[], [""], ["ACGT"], ["", targets[0][:200]], ["N" * 200], ["A" * 200, "ACGT" * 60], [targets[0][:6000]]]
    qs += [[targets[i][:n]] for i in range(9) for n in (900, 1030, 3000)] + [[t[:400] for t in targets[:9]]]
    return qs


def _reads(qs):
    mates = [x for q in qs for x in q]
    qoffs = np.zeros(len(qs) + 1, np.uint32)
    qoffs[1:] = np.cumsum([len(q) for q in qs])
    return u8("".join(mates)), offsets([len(x) for x in mates]), qoffs


def _check(mc, db, odb, parent, taxon, qs, m, with_cands, sizes=(0, 1100, 33000), **cp):
    """The queries as they are (few: one CTA per query) and repeated until
    there are as many as the sort path and the lane-wide lookup start at."""
    import torch
    want = odb.classify(parent, taxon, *_reads(qs), max_candidates=m, with_cands=True, n_threads=8, **cp)
    for size in sizes:
        reps = max(1, -(-size // len(qs)))
        reads, roffs, qoffs = _reads(qs * reps)
        n = len(qoffs) - 1
        cands = torch.zeros(n * m * 4, dtype=torch.int32, device="cuda") if with_cands else None
        got = db.classify(dev(reads), dev(roffs), dev(qoffs), cands=cands, max_candidates=m, **cp)
        mc.mc_classify_status(db.handle)
        for g, o in zip(got, want[:3]):
            bad = np.nonzero(host_u32(g) != np.tile(o, reps))[0]
            assert len(bad) == 0, (size, bad[:10])
        if with_cands:
            assert (host_u32(cands).reshape(n, m, 4) == np.tile(want[3], (reps, 1, 1))).all()


@pytest.fixture(scope="module")
def narrow(mc):
    rng = random.Random(77)
    targets, unit = _targets(rng)
    qs = _queries(rng, targets, unit)
    seq, goffs = "".join(targets), offsets([len(t) for t in targets])
    n = len(targets)
    parent = np.concatenate([[0], np.zeros(9, np.uint32), 1 + np.arange(n) % 9]).astype(np.uint32)
    taxon = np.arange(10, 10 + n, dtype=np.uint32)
    db = gpu_build(mc, u8(seq), goffs, parent, taxon, **P)
    yield db, oracle.DB(seq, goffs, **P), parent, taxon, qs
    db.free()


@pytest.mark.parametrize("with_cands", [False, True])
@pytest.mark.parametrize("m,hits_min,band,max_insert", [(4, 4, 10, 0), (4, 4, 10, 390), (2, 1, 0, 1000), (8, 1, 60, 0),
                                                        (8, 3, 100, 390), (1, 0, 10, 60000), (3, 200, 25, 113)])
def test_filtered_scores_equal_oracle(mc, narrow, m, hits_min, band, max_insert, with_cands):
    db, odb, parent, taxon, qs = narrow
    _check(mc, db, odb, parent, taxon, qs, m, with_cands, hits_min=hits_min, lca_band_pct=band, max_insert=max_insert)


@pytest.mark.parametrize("copies", [4, 5, 16, 17, 32, 33, 64, 65, 128, 129])
def test_class_edges(mc, copies):
    """`copies` targets with the read's 16 features each, and as many that
    share a quarter of them: 16 * copies locations and some, around 64, 256,
    512, 1024 and 2048."""
    rng = random.Random(copies)
    unit = _rand(rng, 128)
    targets = [unit for _ in range(copies)] + [_mutated(rng, unit, 0.05) + _rand(rng, 50) for _ in range(copies // 4)]
    seq, goffs = "".join(targets), offsets([len(t) for t in targets])
    n = len(targets)
    parent, taxon = np.zeros(n + 1, np.uint32), np.arange(1, n + 1, dtype=np.uint32)
    db = gpu_build(mc, u8(seq), goffs, parent, taxon, **P)
    try:
        qs = [[unit], [unit[:60]], [unit, unit[:100]], [_mutated(rng, unit, 0.03)]] * 9
        for with_cands in (False, True):
            _check(mc, db, oracle.DB(seq, goffs, **P), parent, taxon, qs, 4, with_cands, sizes=(0, 1100), hits_min=1,
                   lca_band_pct=10, max_insert=0)
    finally:
        db.free()


def test_wide_locations(mc):
    """64-bit locations: ids that do not fit 32 bits together."""
    import synth
    rng = random.Random(78)
    targets, unit = _targets(rng)
    qs = _queries(rng, targets, unit)
    big, big_o = synth.iid_genomes(17, [7_500_000])
    small, small_o = synth.iid_genomes(18, [24] * ((1 << 17) + 1), stream_base=0xD000000000)
    own = u8("".join(targets))
    genomes = np.concatenate([own, small, big])
    lens = np.concatenate([[len(t) for t in targets], np.diff(small_o), np.diff(big_o)])
    goffs = offsets(lens)
    n = len(lens)
    parent = np.concatenate([[0], np.zeros(64, np.uint32), 1 + np.arange(n) % 64]).astype(np.uint32)
    taxon = np.arange(65, 65 + n, dtype=np.uint32)
    db = gpu_build(mc, genomes, goffs, parent, taxon, **P)
    try:
        assert db.stats()["loc_bytes"] == 8
        odb = oracle.DB(genomes, goffs, **P)
        for m, band, ins, with_cands in [(4, 10, 390, False), (8, 50, 0, True), (4, 100, 1000, False)]:
            _check(mc, db, odb, parent, taxon, qs, m, with_cands, hits_min=2, lca_band_pct=band, max_insert=ins)
    finally:
        db.free()


def test_few_queries_in_every_form(mc, narrow):
    """Launches at and around the number of queries that go straight to one
    CTA each: several batches at once, a plan, and the allocation-free call
    (which has fewer CTAs)."""
    import torch
    db, odb, parent, taxon, qs = narrow
    cls = dict(max_candidates=4, hits_min=2, lca_band_pct=20, max_insert=390)
    cp = mc.classify_params(**cls)
    for sizes in ([7, 0, 1, 30], [511, 1], [300, 213], [1]):
        cuts = np.cumsum([0, *sizes])
        parts = [(qs * 2)[a:b] for a, b in zip(cuts[:-1], cuts[1:])]
        plan = mc.Plan(db.handle, cp, max_batches=len(parts), max_queries=int(cuts[-1]))
        try:
            arrs, outs, keep = [], [], []
            for part in parts:
                reads, roffs, qoffs = _reads(part)
                dv = [dev(reads) if len(reads) else torch.zeros(16, dtype=torch.uint8, device="cuda"), dev(roffs), dev(qoffs)]
                out = [torch.full((max(1, len(part)),), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
                arrs.append(mc.batch(len(roffs) - 1, *dv, *out))
                outs.append(out)
                keep.append(dv)
            for run in (lambda: mc.mc_classify_batches(db.handle, cp, arrs), lambda: plan.run(arrs)):
                for out in outs:
                    for o in out:
                        o.fill_(-7)
                run()
                mc.mc_classify_status(db.handle)
                for part, out in zip(parts, outs):
                    if part:
                        want = odb.classify(parent, taxon, *_reads(part), n_threads=8, **cls)
                        for g, o in zip(out, want):
                            assert (host_u32(g) == o).all()
        finally:
            plan.free()
    for n in (1, 16, 17, 300):
        reads, roffs, qoffs = _reads(qs[:n])
        out = [torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
        mc.mc_classify_noalloc(db.handle, cp, len(roffs) - 1, dev(reads), dev(roffs), n, dev(qoffs), *out)
        mc.mc_classify_status(db.handle)
        want = odb.classify(parent, taxon, reads, roffs, qoffs, n_threads=8, **cls)
        for g, o in zip(out, want):
            assert (host_u32(g) == o).all()

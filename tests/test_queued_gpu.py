"""Queries that the tuning leaves to the medium path: those that a warp can
sort are sorted by warps, the rest go to a CTA each.  Location counts around
the lines, few and many of them, against the oracle."""
import random

import numpy as np
import pytest

import oracle
import test_sort_filter_gpu as sf
from gpu_helpers import dev, gpu_build, gpu_classify, offsets, u8

pytestmark = pytest.mark.gpu
TUNINGS = [dict(sort_max=256), dict(sort_max=512), dict(score_mode=2), dict(score_mode=2, hist_slots=256),
           dict(wide_keys=1, hist_slots=256)]


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


@pytest.mark.parametrize("t", TUNINGS, ids=lambda t: "-".join(f"{k}{v}" for k, v in t.items()))
@pytest.mark.parametrize("copies", [17, 33, 63, 64, 65, 130])
def test_queued_queries(mc, copies, t):
    """16 * copies locations a read and some: 272 to more than 2,048."""
    rng = random.Random(copies)
    unit = sf._rand(rng, 128)
    targets = [unit] * copies + [sf._mutated(rng, unit, 0.05) + sf._rand(rng, 50) for _ in range(copies // 8)]
    targets += [sf._rand(rng, 3000)]
    seq, goffs = "".join(targets), offsets([len(x) for x in targets])
    n = len(targets)
    parent, taxon = np.zeros(n + 1, np.uint32), np.arange(1, n + 1, dtype=np.uint32)
    db = gpu_build(mc, u8(seq), goffs, parent, taxon, **sf.P)
    try:
        mc.mc_db_set_tuning(db.handle, mc.tuning(**t))
        odb = oracle.DB(seq, goffs, **sf.P)
        qs = [[unit], [targets[-1][200:350]], [unit[:60]], [unit, unit[:100]], [sf._mutated(rng, unit, 0.03)]] * 9
        mc.mc_trace_report()
        mc.mc_trace_enable(True)
        try:
            for m, band, with_cands in ((4, 10, False), (8, 50, True), (2, 100, False)):
                sf._check(mc, db, odb, parent, taxon, qs, m, with_cands, sizes=(600, 17_000), hits_min=1,
                          lca_band_pct=band, max_insert=0)
        finally:
            mc.mc_trace_enable(False)
        assert mc.mc_trace_report()["classify_queued"][0] == 6
        # a counting call counts them all
        cls = dict(hits_min=1, lca_band_pct=10, max_insert=0)
        reads, roffs, qoffs = sf._reads(qs)
        ctr = gpu_classify(mc, db, reads, roffs, qoffs, **cls)[-1]
        st = odb.classify(parent, taxon, reads, roffs, qoffs, max_candidates=4, with_stats=True, n_threads=8, **cls)[3]
        assert [int(ctr[i]) for i in range(3)] == [int(st[:, i].sum()) for i in range(3)]
    finally:
        db.free()


@pytest.mark.parametrize("t", TUNINGS[:4], ids=lambda t: "-".join(f"{k}{v}" for k, v in t.items()))
def test_reads_of_every_kind(mc, t):
    rng = random.Random(77)
    targets, unit = sf._targets(rng)
    qs = sf._queries(rng, targets, unit)
    seq, goffs = "".join(targets), offsets([len(x) for x in targets])
    n = len(targets)
    parent = np.concatenate([[0], np.zeros(9, np.uint32), 1 + np.arange(n) % 9]).astype(np.uint32)
    taxon = np.arange(10, 10 + n, dtype=np.uint32)
    db = gpu_build(mc, u8(seq), goffs, parent, taxon, **sf.P)
    try:
        mc.mc_db_set_tuning(db.handle, mc.tuning(**t))
        for with_cands in (False, True):
            sf._check(mc, db, oracle.DB(seq, goffs, **sf.P), parent, taxon, qs, 4, with_cands, sizes=(0, 1100, 17_000),
                      hits_min=2, lca_band_pct=10, max_insert=390)
    finally:
        db.free()

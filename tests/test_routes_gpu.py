"""Instances of the classification kernels that few inputs reach, against the
oracle: the lane-wide lookup with other database parameters and launch
shapes, the sort path at each largest size class, and calls without counters
on the workloads whose tests count (a counting call drops no location before
the sort and never takes the one-kernel route).  Integer work: equality."""
import random

import numpy as np
import pytest

import oracle
import synth
import test_sort_filter_gpu as sf
from gpu_helpers import dev, gpu_build, host_u32, offsets, u8

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


def _windows(length, k, stride):
    return 0 if length < k else (length - k) // stride + 1


# k < 16, s < 16, and each window class (up to 128, 256 and 512 bases)
@pytest.mark.parametrize("p", [dict(k=12, sketch_size=8, window_len=64, window_stride=40),
                               dict(k=4, sketch_size=16, window_len=128, window_stride=125),
                               dict(k=11, sketch_size=7, window_len=200, window_stride=150),
                               dict(k=16, sketch_size=16, window_len=256, window_stride=241),
                               dict(k=15, sketch_size=15, window_len=257, window_stride=243),
                               dict(k=16, sketch_size=9, window_len=512, window_stride=300),
                               dict(k=13, sketch_size=1, window_len=400, window_stride=120)],
                         ids=lambda p: "k{k}-s{sketch_size}-w{window_len}".format(**p))
def test_lane_lookup_of_other_databases(mc, p):
    rng = random.Random(p["window_len"])
    targets, unit = sf._targets(rng)
    k, stride = p["k"], p["window_stride"]
    qs = sf._queries(rng, targets, unit)
    # as many windows as the lane-wide lookup takes (8) and one more, short
    # periods (exact reselection), and a run of invalid bases
    most = k + 8 * stride - 1
    qs += [[t[: min(n, 1024)]] for t in targets[:8] for n in (most, most + 1, most // 2)]
    qs += [[("ACGTTGCA" * 200)[a: a + 400]] for a in range(8)] + [["ACG" * 130, targets[1][:200]], ["A" * 500]]
    qs += [[targets[2][:150] + "N" * 90 + targets[2][240:600]]]
    counts = [sum(_windows(len(x), k, stride) for x in q) for q in qs]
    assert max(c for q, c in zip(qs, counts) if sum(map(len, q)) <= 1024) >= min(8, _windows(1024, k, stride))
    qs = [q for q, c in zip(qs, counts) if c <= 64]  # a query's limit
    seq, goffs = u8("".join(targets)), offsets([len(t) for t in targets])
    n = len(targets)
    parent = np.concatenate([[0], np.zeros(9, np.uint32), 1 + np.arange(n) % 9]).astype(np.uint32)
    taxon = np.arange(10, 10 + n, dtype=np.uint32)
    p = dict(p, bucket_cap=254)
    db = gpu_build(mc, seq, goffs, parent, taxon, **p)
    try:
        odb = oracle.DB(seq, goffs, **p)
        for t in (dict(), dict(probe_batch=4), dict(probe_batch=8, lookup_warps=4), dict(probe_batch=2, lookup_warps=4)):
            mc.mc_db_set_tuning(db.handle, mc.tuning(**t))
            sf._check(mc, db, odb, parent, taxon, qs, 4, not t, sizes=(16_384,), hits_min=1, lca_band_pct=10,
                      max_insert=390)
    finally:
        db.free()


@pytest.mark.parametrize("sort_max", [256, 512, 1024, 2048])
@pytest.mark.parametrize("copies", [15, 16, 17, 32, 64, 65, 100, 127, 128, 129])
def test_sort_classes(mc, copies, sort_max):
    """16 * copies locations a read, all of them equally good (more than 256
    are left to sort), and as many with some of less weight; every class up
    to sort_max is the one that takes them."""
    import torch
    rng = random.Random(1000 + copies)
    unit = sf._rand(rng, 128)
    targets = [unit] * copies + [sf._mutated(rng, unit, 0.05) + sf._rand(rng, 50) for _ in range(copies // 3)]
    seq, goffs = "".join(targets), offsets([len(t) for t in targets])
    n = len(targets)
    parent, taxon = np.zeros(n + 1, np.uint32), np.arange(1, n + 1, dtype=np.uint32)
    db = gpu_build(mc, u8(seq), goffs, parent, taxon, **sf.P)
    try:
        mc.mc_db_set_tuning(db.handle, mc.tuning(sort_max=sort_max))
        odb = oracle.DB(seq, goffs, **sf.P)
        qs = [[unit], [unit[:60]], [unit, unit[:100]], [sf._mutated(rng, unit, 0.03)], [unit[:40], unit[90:]]] * 9
        for m, band, with_cands in ((4, 10, False), (8, 50, True), (2, 100, False)):
            sf._check(mc, db, odb, parent, taxon, qs, m, with_cands, sizes=(1100,), hits_min=1, lca_band_pct=band,
                      max_insert=0)
        reads, roffs, qoffs = sf._reads(qs)
        ctr = torch.zeros(mc.MC_DEBUG_COUNTERS, dtype=torch.int64, device="cuda")
        cls = dict(max_candidates=4, hits_min=1, lca_band_pct=10, max_insert=0)
        db.classify(dev(reads), dev(roffs), dev(qoffs), counters=ctr, **cls)
        mc.mc_classify_status(db.handle)
        locs = odb.classify(parent, taxon, reads, roffs, qoffs, with_stats=True, n_threads=8, **cls)[3][:, 1]
        taken = [int(ctr[7 + 3 * c]) for c in (1, 2, 3, 6)]
        edges = [0, 256, 512, 1024, 2048]
        for c, (lo, hi) in enumerate(zip(edges[:-1], edges[1:])):
            within = int(((locs > lo) & (locs <= hi)).sum()) + (int((locs == 0).sum()) if c == 0 else 0)
            assert taken[c] == (within if hi <= sort_max else 0)
    finally:
        db.free()


def _tiny():
    w = synth.tiny_workload(n_reads=3000, n_decoys=300)
    return w, w.db_params, w.cls_params


def _genera():
    w = synth.mid_workload(seed=1001, n_pairs=18_000, n_families=1, genera_per_family=3, len_scale=0.05, held_genera=1,
                           held_per_genus=3)
    return w, w.db_params, w.cls_params


def _short_windows():
    w = synth.mid_workload(seed=3, n_pairs=2000, n_families=1, genera_per_family=2, len_scale=0.02, held_genera=0)
    return (w, dict(k=12, sketch_size=8, window_len=64, window_stride=40, bucket_cap=20),
            dict(max_candidates=4, hits_min=2, lca_band_pct=20, max_insert=300))


def _repeats():
    w = synth.large_workload(seed=91, n_pairs=3000, n_families=1, genera_per_family=2, n_euk=4, len_scale=0.02,
                             euk_scale=0.03)
    return w, dict(w.db_params, bucket_cap=254), w.cls_params


def _wide_sketch():
    w = synth.tiny_workload(n_reads=3000, n_decoys=300)
    return w, dict(w.db_params, sketch_size=32), w.cls_params


@pytest.mark.parametrize("workload", [_tiny, _genera, _short_windows, _repeats, _wide_sketch], ids=lambda f: f.__name__)
@pytest.mark.parametrize("loaded", [False, True])
def test_calls_without_counters(mc, tmp_path, workload, loaded):
    import torch
    w, p, cls = workload()
    db = gpu_build(mc, w.genomes, w.goffs, w.parent, w.taxon_of_target, **p)
    if loaded:
        db.save(str(tmp_path / "db"))
        db.free()
        db = mc.Database.load(str(tmp_path / "db"))
    try:
        odb = oracle.DB(w.genomes, w.goffs, **p)
        n = len(w.qoffs) - 1
        for part in (n, 512, 40):  # the sort path, the one-kernel route
            qoffs = w.qoffs[: part + 1]
            want = odb.classify(w.parent, w.taxon_of_target, w.reads, w.roffs, qoffs, n_threads=8, with_cands=True,
                                **cls)
            for with_cands in (False, True):
                m = cls["max_candidates"]
                cands = torch.zeros(part * m * 4, dtype=torch.int32, device="cuda") if with_cands else None
                got = db.classify(dev(w.reads), dev(w.roffs), dev(qoffs), cands=cands, **cls)
                mc.mc_classify_status(db.handle)
                for g, o in zip(got, want[:3]):
                    assert (host_u32(g) == o).all()
                if with_cands:
                    assert (host_u32(cands).reshape(part, m, 4) == want[3]).all()
    finally:
        db.free()

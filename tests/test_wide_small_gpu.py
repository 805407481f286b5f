"""Small launches against a database of 64-bit locations: the one-kernel
route, one size class for all, every class, counting calls.  Equal to the
oracle, and as many kernels as the launch needs."""
import random

import numpy as np
import pytest

import oracle
import synth
import test_sort_filter_gpu as sf
from gpu_helpers import dev, gpu_build, gpu_classify, host_u32, offsets, u8

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


@pytest.fixture(scope="module")
def wide(mc):
    rng = random.Random(80)
    targets, unit = sf._targets(rng)
    qs = sf._queries(rng, targets, unit)
    big, big_o = synth.iid_genomes(17, [7_500_000])
    small, small_o = synth.iid_genomes(18, [24] * ((1 << 17) + 1), stream_base=0xD000000000)
    genomes = np.concatenate([u8("".join(targets)), small, big])
    goffs = offsets(np.concatenate([[len(t) for t in targets], np.diff(small_o), np.diff(big_o)]))
    n = len(goffs) - 1
    parent = np.concatenate([[0], np.zeros(64, np.uint32), 1 + np.arange(n) % 64]).astype(np.uint32)
    taxon = np.arange(65, 65 + n, dtype=np.uint32)
    db = gpu_build(mc, genomes, goffs, parent, taxon, **sf.P)
    assert db.stats()["loc_bytes"] == 8
    yield db, oracle.DB(genomes, goffs, **sf.P), parent, taxon, qs
    db.free()


CLS = dict(hits_min=2, lca_band_pct=20, max_insert=390)


# the one-kernel route up to 304 queries (two CTAs on each of 152 SMs); the largest class alone (lookup,
# class, medium, large) up to two queries for each of its resident warps; all
# three classes
@pytest.mark.parametrize("n,kernels", [(1, 1), (40, 1), (304, 1), (305, 4), (512, 4), (1500, 4), (9000, 6),
                                       (20_000, 6)])
@pytest.mark.parametrize("m,with_cands", [(4, False), (8, True)])
def test_small_launches(mc, wide, n, kernels, m, with_cands):
    import torch
    db, odb, parent, taxon, qs = wide
    reads, roffs, qoffs = sf._reads([qs[i % len(qs)] for i in range(n)])
    ins = [dev(reads) if len(reads) else torch.zeros(16, dtype=torch.uint8, device="cuda"), dev(roffs), dev(qoffs)]
    cands = torch.zeros(n * m * 4, dtype=torch.int32, device="cuda") if with_cands else None
    before = mc.mc_kernel_launches()
    got = db.classify(*ins, cands=cands, max_candidates=m, **CLS)
    launched = mc.mc_kernel_launches() - before
    mc.mc_classify_status(db.handle)
    want = odb.classify(parent, taxon, *sf._reads(qs), max_candidates=m, with_cands=True, n_threads=8, **CLS)
    for g, o in zip(got, want):
        assert (host_u32(g) == np.resize(o, n)).all()
    if with_cands:
        assert (host_u32(cands).reshape(n, m, 4) == want[3][np.arange(n) % len(qs)]).all()
    assert launched == kernels


@pytest.mark.parametrize("n", [8, 9, 16, 17, 600])
def test_allocation_free(mc, wide, n):
    import torch
    db, odb, parent, taxon, qs = wide
    reads, roffs, qoffs = sf._reads(qs[:n])
    out = [torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
    mc.mc_classify_noalloc(db.handle, mc.classify_params(**CLS), len(roffs) - 1, dev(reads), dev(roffs), n, dev(qoffs),
                           *out)
    mc.mc_classify_status(db.handle)
    want = odb.classify(parent, taxon, reads, roffs, qoffs, max_candidates=4, n_threads=8, **CLS)
    for g, o in zip(out, want):
        assert (host_u32(g) == o).all()


def test_counting_call(mc, wide):
    """Counts every distinct location; the histogram kernel takes what it holds."""
    db, odb, parent, taxon, qs = wide
    reads, roffs, qoffs = sf._reads(qs)
    got = gpu_classify(mc, db, reads, roffs, qoffs, **CLS)
    want = odb.classify(parent, taxon, reads, roffs, qoffs, max_candidates=4, with_stats=True, n_threads=8, **CLS)
    for g, o in zip(got[:3], want[:3]):
        assert (g == o).all()
    ctr = got[-1]
    assert [int(ctr[i]) for i in range(3)] == [int(want[3][:, i].sum()) for i in range(3)]
    bases = np.array([sum(map(len, q)) for q in qs])
    assert int(ctr[7]) >= int(((want[3][:, 1] <= 256) & (bases <= 900)).sum()) > 200  # it holds 384 distinct


def test_autotuner_times_each_shape_once(mc, wide):
    """64-bit locations have no size class beyond 1,024."""
    import torch
    db, odb, parent, taxon, qs = wide
    reads, roffs, qoffs = sf._reads(qs)
    out = [torch.zeros(len(qs), dtype=torch.int32, device="cuda") for _ in range(3)]
    b = mc.batch(len(roffs) - 1, dev(reads), dev(roffs), dev(qoffs), *out)
    cp = mc.classify_params(**CLS)
    best, rec = mc.mc_autotune(db.handle, cp, [b], reps=1)
    assert len(rec) == 6 + 18 + 3
    mc.mc_classify_batches(db.handle, cp, [b], best)
    mc.mc_classify_status(db.handle)
    want = odb.classify(parent, taxon, reads, roffs, qoffs, max_candidates=4, n_threads=8, **CLS)
    for g, o in zip(out, want):
        assert (host_u32(g) == o).all()

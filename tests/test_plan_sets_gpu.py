"""Plans run with far fewer queries than they hold: such a run launches what
a call of its own size does, not what the plan's capacity would, and gives
the same results.  Sizes around the lines between the kernels."""
import random

import numpy as np
import pytest

import oracle
import test_sort_filter_gpu as sf
from gpu_helpers import dev, gpu_build, host_u32, offsets, u8

pytestmark = pytest.mark.gpu
CAPACITY = 60_000
CLS = dict(max_candidates=4, hits_min=2, lca_band_pct=20, max_insert=390)


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


@pytest.fixture(scope="module")
def setup(mc):
    rng = random.Random(79)
    targets, unit = sf._targets(rng)
    qs = sf._queries(rng, targets, unit)
    seq, goffs = u8("".join(targets)), offsets([len(t) for t in targets])
    n = len(targets)
    parent = np.concatenate([[0], np.zeros(9, np.uint32), 1 + np.arange(n) % 9]).astype(np.uint32)
    taxon = np.arange(10, 10 + n, dtype=np.uint32)
    db = gpu_build(mc, seq[: goffs[-2]], goffs[:-1], parent, taxon[:-1], **sf.P)
    plan = mc.Plan(db.handle, mc.classify_params(**CLS), max_batches=3, max_queries=CAPACITY)
    yield db, plan, qs, (seq, goffs, parent, taxon)
    plan.free()
    db.free()


def _set(mc, qs, n):
    """n queries (qs over and over) as three batches of uneven size."""
    import torch
    cuts = [0, n // 7, n - n // 3, n]
    arrs, outs, keep = [], [], []
    for a, b in zip(cuts[:-1], cuts[1:]):
        part = [qs[i % len(qs)] for i in range(a, b)]
        reads, roffs, qoffs = sf._reads(part)
        dv = [dev(reads) if len(reads) else torch.zeros(16, dtype=torch.uint8, device="cuda"), dev(roffs), dev(qoffs)]
        out = [torch.full((max(1, len(part)),), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
        arrs.append(mc.batch(len(roffs) - 1, *dv, *out))
        outs.append((len(part), out))
        keep.append(dv)
    return arrs, outs, keep


def _run(mc, db, run, outs):
    """What the run gives, and the kernels it launches."""
    for _, out in outs:
        for o in out:
            o.fill_(-7)
    before = mc.mc_kernel_launches()
    run()
    launched = mc.mc_kernel_launches() - before
    mc.mc_classify_status(db.handle)
    return [np.concatenate([host_u32(out[i])[:k] for k, out in outs]) for i in range(3)], launched


# the last size comes back to a set that was captured before
@pytest.mark.parametrize("n", [1, 16, 512, 513, 2000, 16_383, 16_384, 20_000, CAPACITY, 16])
def test_run_of_any_size_equals_a_call_of_that_size(mc, setup, n):
    db, plan, qs, (seq, goffs, parent, taxon) = setup
    arrs, outs, keep = _set(mc, qs, n)
    cp = mc.classify_params(**CLS)
    got, launched = _run(mc, db, lambda: plan.run(arrs), outs)
    call, launched_by_call = _run(mc, db, lambda: mc.mc_classify_batches(db.handle, cp, arrs), outs)
    assert launched == launched_by_call
    odb = oracle.DB(seq[: goffs[-2]], goffs[:-1], **sf.P)
    want = odb.classify(parent, taxon[:-1], *sf._reads(qs), n_threads=8, **CLS)
    for g, c, o in zip(got, call, want):
        o = np.resize(o, n)
        assert (g == o).all() and (c == o).all()


def test_empty_run(mc, setup):
    db, plan, qs, _ = setup
    plan.run([])
    mc.mc_classify_status(db.handle)


def test_every_set_follows_an_extension(mc, setup):
    """Sets captured before an extension of the database serve the extended one."""
    db, plan, qs, (seq, goffs, parent, taxon) = setup
    lo = int(goffs[-2])
    for n in (16, 2000, CAPACITY):  # captured
        plan.run(_set(mc, qs, n)[0])
    mc.mc_classify_status(db.handle)
    db.add_targets(dev(seq[lo:]), dev((goffs[-2:] - goffs[-2]).astype(np.uint64)), taxon[-1:])
    db.finalize()
    more = [[x] for x in ("".join(map(chr, seq[lo + 100 * i: lo + 100 * i + 120])) for i in range(15))] + qs
    want = oracle.DB(seq, goffs, **sf.P).classify(parent, taxon, *sf._reads(more), n_threads=8, **CLS)
    assert (want[2][:15] == len(taxon) - 1).any()
    for n in (16, 2000, CAPACITY):
        arrs, outs, keep = _set(mc, more, n)
        got, _ = _run(mc, db, lambda: plan.run(arrs), outs)
        for g, o in zip(got, want):
            assert (g == np.resize(o, n)).all()

"""Calls of several host threads that launch the same kernel with different
shared-memory sizes: none is refused, and each gives what it gives alone."""
import threading

import pytest

import oracle
import synth
from gpu_helpers import dev, gpu_build, host_u32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2106_08150_gb300 import mc as m
    m.use_torch_allocator()
    return m


def _together(calls):
    """Runs the calls, a thread each; returns what they raised."""
    raised = []

    def run(f):
        try:
            f()
        except Exception as e:  # noqa: BLE001
            raised.append(e)

    threads = [threading.Thread(target=run, args=(f,)) for f in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return raised


def test_sketches_with_other_windows(mc):
    """Windows of 128 and of 64 bases: one kernel, 34 and 30 KB."""
    import torch
    calls, outs = [], []
    for w, stride in ((128, 113), (64, 10)):
        genomes, offs = synth.iid_genomes(5, [4000])
        prm = mc.db_params(window_len=w, window_stride=stride)
        seq, o = dev(genomes), dev(offs)
        win = torch.zeros(2, dtype=torch.int64, device="cuda")
        mc.mc_window_offsets(prm, 1, o, win)
        n_win = int(win[-1])
        sketch = torch.zeros(n_win * 16, dtype=torch.int32, device="cuda")
        counts = torch.zeros(n_win, dtype=torch.int32, device="cuda")
        stream = torch.cuda.Stream()

        def sketch_many(prm=prm, seq=seq, o=o, win=win, n_win=n_win, sketch=sketch, counts=counts, stream=stream):
            for _ in range(20_000):
                mc.mc_sketch(prm, 1, seq, o, win, n_win, sketch, counts, stream=stream)
            stream.synchronize()

        mc.mc_sketch(prm, 1, seq, o, win, n_win, sketch, counts)
        torch.cuda.synchronize()
        outs.append((sketch, sketch.clone(), counts, counts.clone()))
        calls.append(sketch_many)
    assert _together(calls) == []
    for sketch, want, counts, want_counts in outs:
        assert torch.equal(sketch, want) and torch.equal(counts, want_counts)


def test_classify_with_other_sketch_sizes(mc):
    """Databases of sketch size 16 and 8, whose bucket lists take different
    room in the same lookup and scoring kernels."""
    import torch
    w = synth.tiny_workload(n_reads=700, n_decoys=70)
    calls, checks = [], []
    for s, mode in ((16, 1), (8, 1), (16, 2), (8, 2)):
        p = dict(w.db_params, sketch_size=s)
        db = gpu_build(mc, w.genomes, w.goffs, w.parent, w.taxon_of_target, **p)
        mc.mc_db_set_tuning(db.handle, mc.tuning(score_mode=mode))
        want = oracle.DB(w.genomes, w.goffs, **p).classify(w.parent, w.taxon_of_target, w.reads, w.roffs, w.qoffs,
                                                           n_threads=8, **w.cls_params)
        cp = mc.classify_params(**w.cls_params)
        n, ins = len(w.qoffs) - 1, [dev(w.reads), dev(w.roffs), dev(w.qoffs)]
        out = [torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)]

        def classify_many(db=db, cp=cp, n=n, ins=ins, out=out):
            stream = torch.cuda.Stream()
            for _ in range(1500):
                mc.mc_classify(db.handle, cp, len(w.roffs) - 1, ins[0], ins[1], n, ins[2], *out, stream=stream)
            stream.synchronize()

        calls.append(classify_many)
        checks.append((db, out, want))
    try:
        torch.cuda.synchronize()
        assert _together(calls) == []
        for db, out, want in checks:
            for g, o in zip(out, want):
                assert (host_u32(g) == o).all()
    finally:
        for db, _, _ in checks:
            db.free()

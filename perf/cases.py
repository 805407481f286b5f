"""The work that users of the library have it do, as a list of measurable
cases: classifying read sets of every size against a resident database,
building a database and classifying against it in one go, growing a
database while it is used, partitioned databases, and serving jobs.

Sizes and recipes follow the library's own configurations (`synth/`,
`tests/`, `bench.py`): genera of related genomes, repeat-rich genomes with
satellite arrays, draft assemblies of many scaffolds; 2x150 bp pairs,
single-end reads, mixed lengths 50-300, reads of a few kbp.  Inputs are
drawn on the device from the seed alone.

Every output is a whole number (taxon ids, hit counts, target ids,
candidate lists, database counters).
"""
import math
import random

import torch

# ---------------------------------------------------------------- recipes
# Databases.  genera x species x strains related genomes (median length
# `mbp`), n_rep repeat-rich genomes, n_scaf scaffolds of a draft assembly
# (with n_chr chromosomes of 8 Mbp and more): the last kind has target and
# window ids that do not fit 32 bits together.
TINY = dict(genera=2, species=2, strains=2, mbp=0.2, n_rep=0, rep_mbp=0.0, n_scaf=0, n_chr=0)
SMALL = dict(genera=20, species=5, strains=2, mbp=0.3, n_rep=0, rep_mbp=0.0, n_scaf=0, n_chr=0)
MID = dict(genera=100, species=5, strains=2, mbp=3.0, n_rep=0, rep_mbp=0.0, n_scaf=0, n_chr=0)
LARGE = dict(genera=980, species=5, strains=2, mbp=1.1, n_rep=200, rep_mbp=12.5, n_scaf=0, n_chr=0)
REPEATS = dict(genera=4, species=5, strains=2, mbp=1.1, n_rep=24, rep_mbp=12.5, n_scaf=0, n_chr=0)
DRAFT = dict(genera=0, species=0, strains=0, mbp=0.0, n_rep=0, rep_mbp=0.0, n_scaf=140_000, n_chr=12)
GROWN = dict(genera=60, species=5, strains=2, mbp=1.1, n_rep=0, rep_mbp=0.0, n_scaf=0, n_chr=0)

# Database parameters: the paper's defaults (window overlap k - 1).
DEFAULT = dict(k=16, sketch=16, window=128, stride=113, cap=254)
PAPER_127 = dict(k=16, sketch=16, window=127, stride=112, cap=254)
SHORT = dict(k=12, sketch=8, window=64, stride=40, cap=20)

# Read sets: lengths uniform in [lo, hi] (both mates alike), `paired` share
# of pairs, fragments N(1.5 * length + 75, 10%).
PAIRS_150 = dict(lo=150, hi=150, paired=1.0, max_insert=390)
PAIRS_100 = dict(lo=100, hi=100, paired=1.0, max_insert=300)
MIXED = dict(lo=50, hi=300, paired=0.5, max_insert=0)
SINGLE_100 = dict(lo=100, hi=100, paired=0.0, max_insert=0)
SINGLE_250 = dict(lo=250, hi=250, paired=0.0, max_insert=0)
LONG = dict(lo=1000, hi=6000, paired=0.0, max_insert=0)


def listed():
    return [
        # an interactive query: a handful of pairs, one call
        dict(name="pairs_16", kind="classify", call="classify", n_q=16, parts=1, **SMALL, **DEFAULT, **PAIRS_150),
        # a request loop: a set of small batches through a CUDA-graph plan
        dict(name="plan_20k", kind="classify", call="plan", n_q=20_000, parts=8, **SMALL, **DEFAULT, **MIXED),
        # a sequencer's read set against the large resident database
        dict(name="pairs_2m_large", kind="classify", call="classify", n_q=2_000_000, parts=1, **LARGE, **DEFAULT,
             **PAIRS_150),
        # many samples at once: batches of uneven size and read length
        dict(name="batches_700k", kind="classify", call="batches", n_q=700_000, parts=64, **MID, **DEFAULT, **MIXED),
        # a database partitioned by target: every part's candidate lists, merged
        dict(name="shards_200k", kind="classify", call="shards", n_q=200_000, parts=2, **GROWN, **DEFAULT,
             **SINGLE_250),
        # amplicons and assembled reads of a few kbp
        dict(name="long_5k", kind="classify", call="classify", n_q=5_000, parts=1, **GROWN, **DEFAULT, **LONG),
        # draft assemblies: many scaffolds, 64-bit locations
        dict(name="draft_300k", kind="classify", call="classify", n_q=300_000, parts=1, **DRAFT, **DEFAULT,
             **PAIRS_100),
        # a small reference set built and queried on the fly
        dict(name="build_tiny", kind="build", n_q=11_000, parts=1, **TINY, **DEFAULT, **SINGLE_100),
        # repeat-rich genomes: capped buckets, satellite arrays
        dict(name="build_repeats", kind="build", n_q=200_000, parts=1, **REPEATS, **PAPER_127, **PAIRS_150),
        # the headline workload: the large reference set built and queried on the fly
        dict(name="build_large", kind="build", n_q=4_000_000, parts=1, **LARGE, **DEFAULT, **PAIRS_150),
        # a database that grows while it is used
        dict(name="grow_4", kind="grow", n_q=50_000, parts=5, **GROWN, **DEFAULT, **PAIRS_150),
        # a served stream of jobs on host buffers
        dict(name="serve_16", kind="serve", n_q=160_000, parts=16, **SMALL, **DEFAULT, **MIXED),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["classify", "classify", "classify", "classify", "build", "build", "grow", "serve"])
    prm = rng.choice([DEFAULT, DEFAULT, PAPER_127, SHORT])
    reads = dict(rng.choice([PAIRS_150, PAIRS_100, MIXED, SINGLE_100, SINGLE_250]))
    if reads["lo"] == reads["hi"]:
        reads["lo"] = reads["hi"] = reads["hi"] + rng.randrange(-17, 18)
    else:
        reads["lo"], reads["hi"] = reads["lo"] + rng.randrange(0, 30), reads["hi"] - rng.randrange(0, 50)
    db = dict(TINY, genera=_log(rng, 2, 200), species=rng.randrange(1, 6), strains=rng.randrange(1, 4),
              mbp=round(math.exp(rng.uniform(math.log(0.2), math.log(1.5))), 3))
    if kind == "classify":
        call = rng.choice(["classify", "classify", "noalloc", "plan", "batches", "shards", "long", "draft"])
        n_q = _log(rng, 1, 700_000)
        parts = 1
        if call == "noalloc":
            n_q = _log(rng, 1, 16_000)
        elif call in ("plan", "batches"):
            parts = rng.randrange(2, 65)
            n_q = max(n_q, parts)
        elif call == "shards":
            parts = rng.randrange(2, 5)
            n_q = min(n_q, 200_000)
        elif call == "long":
            call, reads, n_q = "classify", dict(LONG, lo=500 + rng.randrange(500), hi=1500 + rng.randrange(4500)), \
                _log(rng, 1, 5_000)
            prm = rng.choice([DEFAULT, PAPER_127])  # 64 windows of a query reach 6 kbp with these
        elif call == "draft":
            call, db, prm = "classify", dict(DRAFT, n_scaf=132_000 + rng.randrange(60_000),
                                             n_chr=rng.randrange(2, 13)), rng.choice([DEFAULT, PAPER_127])
            n_q = min(n_q, 300_000)
        return dict(kind=kind, call=call, n_q=n_q, parts=parts, **db, **prm, **reads)
    if kind == "build":
        db["n_rep"], db["rep_mbp"] = rng.choice([(0, 0.0), (rng.randrange(1, 30), round(rng.uniform(2, 14), 2))])
        return dict(kind=kind, n_q=_log(rng, 1_000, 1_000_000), parts=rng.randrange(1, 4), **db, **prm, **reads)
    if kind == "grow":
        db["genera"] = max(8, min(db["genera"], 60))
        return dict(kind=kind, n_q=_log(rng, 1_000, 100_000), parts=rng.randrange(2, 6), **db, **prm, **reads)
    db["genera"] = min(db["genera"], 40)
    return dict(kind=kind, n_q=_log(rng, 2_000, 160_000), parts=rng.randrange(2, 33), **db, **prm, **reads)


# ----------------------------------------------------------------- inputs
def _bases(gen, n, gc):
    """n random bases (ASCII) with the given GC share."""
    g = round(256 * gc / 2)
    lut = torch.tensor([65] * (128 - g) + [67] * g + [71] * g + [84] * (128 - g), dtype=torch.uint8, device="cuda")
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    for a in range(0, n, 1 << 26):
        m = min(1 << 26, n - a)
        r = torch.randint(0, 256, (m,), dtype=torch.uint8, device="cuda", generator=gen)
        out[a:a + m] = lut[r.int()]
    return out


def _new_bases(pos, salt):
    """A base for each position: a function of the position, so that one
    drawn twice gets the same base both times."""
    acgt = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    return acgt[((pos + salt) * 2654435761 >> 13) & 3]


def _mutate(gen, py, flat, n, pos=None):
    """Substitutes n random positions of `flat` (or those given)."""
    if pos is None:
        pos = torch.randint(0, flat.numel(), (n,), device="cuda", generator=gen)
    flat[pos] = _new_bases(pos, py.randrange(1 << 20))


def _genomes(case, gen, py):
    """(bases, host offsets, parent, taxon of each target)."""
    sp, st = case["species"], case["strains"]
    lens = []
    for _ in range(case["genera"]):
        lens += [max(1000, int(case["mbp"] * 1e6 * math.exp(py.gauss(0, 0.5))))] * (sp * st)
    lens += [int(case["rep_mbp"] * 1e6 * py.uniform(0.4, 1.6)) for _ in range(case["n_rep"])]
    lens += [8_000_000 + py.randrange(2_000_000) for _ in range(case["n_chr"])]
    lens += [300 + int(1500 * py.expovariate(1.0)) for _ in range(case["n_scaf"])]
    offs = [0]
    for n in lens:
        offs.append(offs[-1] + n)
    blob = torch.empty(offs[-1], dtype=torch.uint8, device="cuda")
    at = 0
    for g in range(case["genera"]):
        n, root = lens[at], offs[at]
        part = blob[root:root + n * sp * st]
        part.view(sp * st, n).copy_(_bases(gen, n, py.uniform(0.3, 0.7)).expand(sp * st, n))
        for s in range(sp):  # species: 1-5% from the root, the same in all their strains
            m = int(py.uniform(0.01, 0.05) * n)
            pos = torch.randint(0, n, (m,), device="cuda", generator=gen)
            part.view(sp, st, n)[s][:, pos] = _new_bases(pos, py.randrange(1 << 20))
        _mutate(gen, py, part, part.numel() // 1000)  # strains: 0.1%
        at += sp * st
    for _ in range(case["n_rep"]):  # 5 kbp segments: 30% copies of another one, 2% satellite arrays
        n, a = lens[at], offs[at]
        one = _bases(gen, n, py.uniform(0.3, 0.7))
        seg = torch.arange(n, device="cuda") // 5000
        n_seg = n // 5000 + 1
        what = torch.rand(n_seg, device="cuda", generator=gen)
        shift = (torch.rand(n_seg, device="cuda", generator=gen) * max(1, n - 5000)).long()
        src = torch.where(what[seg] < 0.3, shift[seg] + torch.arange(n, device="cuda") % 5000,
                          torch.arange(n, device="cuda"))
        src = torch.where(what[seg] > 0.98, torch.arange(n, device="cuda") % 171, src)
        one = one[src]
        _mutate(gen, py, one, n // 200)
        blob[a:a + n] = one
        at += 1
    if at < len(lens):
        tail = blob[offs[at]:]
        tail.copy_(_bases(gen, tail.numel(), 0.42))
        for _ in range(64):  # gaps of the assembly
            a = py.randrange(max(1, tail.numel() - 1000))
            tail[a:a + py.randrange(1, 1000)] = 78
    n_t = len(lens)
    # root -> genera of ten targets -> targets
    n_g = (n_t + 9) // 10
    parent = [0] * (1 + n_g) + [1 + t // 10 for t in range(n_t)]
    return blob, offs, parent, list(range(1 + n_g, 1 + n_g + n_t))


def _reads(case, gen, py, blob, offs, n_q):
    """(bases, offsets, qoffs): reads of random places of the genomes, 0.5%
    substituted, one in twenty from a species that the genomes do not hold
    (4% substituted), now and then an unread base."""
    off = torch.tensor(offs, device="cuda")
    wide = (off[1:] - off[:-1]) >= 300  # targets long enough to be read from
    tgt = torch.nonzero(wide).reshape(-1)
    if not len(tgt):
        tgt = torch.arange(len(offs) - 1, device="cuda")
    n_pair = int(round(n_q * case["paired"]))
    mates = torch.ones(n_q, dtype=torch.long, device="cuda")
    mates[:n_pair] = 2
    mates = mates[torch.randperm(n_q, device="cuda", generator=gen)]
    qoffs = torch.zeros(n_q + 1, dtype=torch.long, device="cuda")
    qoffs[1:] = mates.cumsum(0)
    ln = torch.randint(case["lo"], case["hi"] + 1, (n_q,), device="cuda", generator=gen)
    weight = None
    if case["n_chr"]:  # of a draft assembly reads come by length
        cum = (off[1:] - off[:-1])[tgt].cumsum(0)
        weight = torch.searchsorted(cum, (torch.rand(n_q, dtype=torch.float64, device="cuda", generator=gen)
                                          * cum[-1]).long())
    t = tgt[weight.clamp_(max=len(tgt) - 1) if weight is not None
            else torch.randint(0, len(tgt), (n_q,), device="cuda", generator=gen)]
    g_len = off[t + 1] - off[t]
    ln = torch.minimum(ln, g_len)
    mean = 1.5 * ln + 75
    frag = torch.where(mates == 2, (mean * (1 + 0.1 * torch.randn(n_q, device="cuda", generator=gen))).long(), ln)
    frag = torch.minimum(torch.maximum(frag, ln), g_len)
    start = off[t] + (torch.rand(n_q, dtype=torch.float64, device="cuda", generator=gen) * (g_len - frag + 1)).long()
    rev = torch.rand(n_q, device="cuda", generator=gen) < 0.5
    # per sequence: first base read, direction, length
    q_of = torch.repeat_interleave(torch.arange(n_q, device="cuda"), mates)
    second = torch.arange(len(q_of), device="cuda") - qoffs[q_of] == 1
    back = rev[q_of] ^ second
    s_len = ln[q_of]
    lo = torch.where(back, start[q_of] + frag[q_of] - 1, start[q_of])
    roffs = torch.zeros(len(q_of) + 1, dtype=torch.long, device="cuda")
    roffs[1:] = s_len.cumsum(0)
    total = int(roffs[-1])
    reads = torch.empty(total, dtype=torch.uint8, device="cuda")
    comp = torch.arange(256, dtype=torch.uint8, device="cuda")
    comp[[65, 67, 71, 84]] = torch.tensor([84, 71, 67, 65], dtype=torch.uint8, device="cuda")
    step = 1 << 18
    for a in range(0, len(q_of), step):
        b = min(a + step, len(q_of))
        r0, r1 = int(roffs[a]), int(roffs[b])
        sid = torch.repeat_interleave(torch.arange(a, b, device="cuda"), s_len[a:b])
        i = torch.arange(r0, r1, device="cuda") - roffs[sid]
        d = back[sid]
        base = blob[lo[sid] + torch.where(d, -i, i)]
        base = torch.where(d, comp[base.int()], base)
        _mutate(gen, py, base, (r1 - r0) // 200)
        foreign = torch.nonzero((torch.rand(r1 - r0, device="cuda", generator=gen) < 0.04) & (q_of[sid] % 20 == 7))
        if len(foreign):
            _mutate(gen, py, base, 0, foreign.reshape(-1))
        base[torch.randint(0, r1 - r0, ((r1 - r0) // 10_000 + 1,), device="cuda", generator=gen)] = 78
        reads[r0:r1] = base
    return reads, roffs, qoffs.int()


def _cut(reads, roffs, qoffs, parts):
    """The read set as `parts` batches of uneven size (the same sizes for
    every seed), each with its own buffers and offsets."""
    n_q = len(qoffs) - 1
    py = random.Random(n_q * 64 + parts)
    share = [math.exp(py.gauss(0, 1)) for _ in range(parts)]
    cut, acc = [0], 0.0
    for x in share[:-1]:
        acc += x
        cut.append(int(n_q * acc / sum(share)))
    cut.append(n_q)
    out = []
    for a, b in zip(cut[:-1], cut[1:]):
        s0, s1 = int(qoffs[a]), int(qoffs[b])
        r0, r1 = int(roffs[s0]), int(roffs[s1])
        seq = reads[r0:r1].clone() if r1 > r0 else torch.zeros(1, dtype=torch.uint8, device="cuda")
        out.append((seq, roffs[s0:s1 + 1] - r0, qoffs[a:b + 1] - s0))
    return out


# ------------------------------------------------------------------- runs
_mc = None


def _lib():
    global _mc
    if _mc is None:
        from paper_2106_08150_gb300 import mc
        mc.use_torch_allocator()
        _mc = mc
    return _mc


def _empty(mc, case, parent):
    import numpy as np
    return mc.Database.create(np.array(parent, dtype=np.uint32), k=case["k"], sketch_size=case["sketch"],
                              window_len=case["window"], window_stride=case["stride"], bucket_cap=case["cap"])


def _split(blob, offs, taxon, parts):
    """The genomes as `parts` runs of whole targets: (bases, offsets, taxa)."""
    import numpy as np
    cut = [len(taxon) * i // parts for i in range(parts + 1)]
    out = []
    for a, b in zip(cut[:-1], cut[1:]):
        seq = blob[offs[a]:offs[b]]
        out.append((seq if seq.data_ptr() % 16 == 0 else seq.clone(),
                    torch.tensor([x - offs[a] for x in offs[a:b + 1]], device="cuda"),
                    np.array(taxon[a:b], dtype=np.uint32)))
    return out


def _counts(db):
    st = db.stats()
    return [st[n] for n in ("n_targets", "n_windows", "n_pairs", "n_keys", "n_locations", "overflow_keys",
                            "dropped_locations")]


class _Serving:
    """A database with its server, released in the right order."""

    def __init__(self, mc, db, cp, max_queries):
        self.db = db
        self.server = mc.Server(db.handle, cp, max_set_queries=max_queries)

    def __del__(self):
        self.server.free()
        self.db.free()


class _Planned:
    """A database with a classification plan, released in the right order."""

    def __init__(self, mc, db, cp, batches, queries):
        self.db = db
        self.plan = mc.Plan(db.handle, cp, max_batches=batches, max_queries=queries)

    def __del__(self):
        self.plan.free()
        self.db.free()


def prepare(case, seed):
    mc = _lib()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    py = random.Random(seed)
    blob, offs, parent, taxon = _genomes(case, gen, py)
    reads, roffs, qoffs = _reads(case, gen, py, blob, offs, case["n_q"])
    cls = dict(max_candidates=4, hits_min=4, lca_band_pct=10, max_insert=case["max_insert"])
    s = dict(case=case, cp=mc.classify_params(**cls), cls=cls, parent=parent)
    if case["kind"] in ("build", "grow"):
        s["targets"] = _split(blob, offs, taxon, case["parts"])
        s["reads"] = (reads, roffs, qoffs)
        return s
    if case["kind"] == "classify" and case["call"] == "shards":
        s["reads"] = (reads, roffs, qoffs)
        s["taxon"] = torch.tensor(taxon, dtype=torch.int32, device="cuda")
        s["shards"], s["base"], prior, at = [], [], [], 0
        for seq, o, tx in _split(blob, offs, taxon, case["parts"]):
            db = _empty(mc, case, parent)
            db.add_targets(seq, o, tx)
            n = mc.mc_db_feature_counts(db.handle)
            keys = torch.empty(max(1, n), dtype=torch.int32, device="cuda")
            counts = torch.empty_like(keys)
            mc.mc_db_feature_counts(db.handle, keys, counts, n)
            mc.mc_db_finalize_after(db.handle, prior)
            prior.append((keys, counts, n))
            s["shards"].append(db)
            s["base"].append(at)
            at += len(tx)
        return s
    db = _empty(mc, case, parent)
    for seq, o, tx in _split(blob, offs, taxon, 1):
        db.add_targets(seq, o, tx)
    db.finalize()
    if case["kind"] == "classify" and case["call"] in ("classify", "noalloc"):
        s["db"], s["reads"] = db, (reads, roffs, qoffs)
        return s
    batches = _cut(reads, roffs, qoffs, case["parts"])
    if case["kind"] == "classify":
        s["batches"], s["cut"], at = batches, [], 0
        s["out"] = [torch.zeros(case["n_q"], dtype=torch.int32, device="cuda") for _ in range(3)]
        for seq, o, q in batches:  # every batch writes its own part of the outputs
            s["cut"].append([x[at:at + len(q) - 1] for x in s["out"]])
            at += len(q) - 1
        if case["call"] == "plan":
            s["planned"] = _Planned(mc, db, s["cp"], len(batches), case["n_q"])
        else:
            s["db"] = db
        return s
    jobs = []
    for seq, o, q in batches:  # host buffers, page-locked as a server's would be
        if len(q) < 2:
            continue
        out = [torch.zeros(len(q) - 1, dtype=torch.int32).pin_memory() for _ in range(3)]
        jobs.append((len(o) - 1, seq.cpu().pin_memory(), o.cpu().pin_memory(), q.cpu().pin_memory(), *out))
    s["jobs"] = jobs
    s["serving"] = _Serving(mc, db, s["cp"], max(1, case["n_q"] // 2))
    return s


def run(s):
    mc, case = _lib(), s["case"]
    if case["kind"] == "build":  # the genomes, in the parts they came in, then the reads
        db = _empty(mc, case, s["parent"])
        for seq, o, tx in s["targets"]:
            db.add_targets(seq, o, tx)
        db.finalize()
        out = db.classify(*s["reads"], **s["cls"])
        counts = _counts(db)
        db.free()
        return {"reads": out, "counts": counts}
    if case["kind"] == "grow":  # queried after every part that came
        db = _empty(mc, case, s["parent"])
        out = []
        for seq, o, tx in s["targets"]:
            db.add_targets(seq, o, tx)
            db.finalize()
            out.append((db.classify(*s["reads"], **s["cls"]), _counts(db)))
        db.free()
        return out
    if case["kind"] == "serve":
        srv = s["serving"].server
        ids = [srv.submit(*j) for j in s["jobs"]]
        for i in ids:
            srv.wait(i)
        return [j[4:] for j in s["jobs"]]
    if case["call"] == "classify":
        return s["db"].classify(*s["reads"], **s["cls"])
    if case["call"] in ("plan", "batches"):
        arr = [mc.batch(len(o) - 1, seq, o, q, *out) for (seq, o, q), out in zip(s["batches"], s["cut"])]
        if case["call"] == "plan":
            s["planned"].plan.run(arr)
        else:
            mc.mc_classify_batches(s["db"].handle, s["cp"], arr)
        return s["out"]
    reads, roffs, qoffs = s["reads"]
    n_q = len(qoffs) - 1
    if case["call"] == "noalloc":
        out = [torch.empty(n_q, dtype=torch.int32, device="cuda") for _ in range(3)]
        mc.mc_classify_noalloc(s["db"].handle, s["cp"], len(roffs) - 1, reads, roffs, n_q, qoffs, *out)
        return out
    m = s["cls"]["max_candidates"]
    lists = []
    for db in s["shards"]:
        c = torch.empty(n_q * m * 4, dtype=torch.int32, device="cuda")
        db.classify(reads, roffs, qoffs, cands=c, **s["cls"])
        lists.append(c)
    out = [torch.empty(n_q, dtype=torch.int32, device="cuda") for _ in range(3)]
    merged = torch.empty(n_q * m * 4, dtype=torch.int32, device="cuda")
    mc.mc_merge_candidates(s["shards"][0].handle, s["cp"], n_q, lists, s["base"], s["taxon"], len(s["taxon"]), *out,
                           merged)
    return [*out, merged]


# ------------------------------------------------------------------- work
def _n_bp(case):
    """Expected bases of the database."""
    g = case["genera"] * case["species"] * case["strains"] * case["mbp"] * 1e6 * math.exp(0.125)
    return g + case["n_rep"] * case["rep_mbp"] * 1e6 + case["n_chr"] * 9e6 + case["n_scaf"] * 1800.0


def work(case):
    """Bytes one pass has to move: the reads and outputs, a 32-byte sector
    of the feature table and one of the locations per feature looked up; a
    build reads its genomes once and writes its pairs' locations and its
    features' table words once.  There is no floating-point work."""
    s, stride = case["sketch"], case["stride"]
    mates = case["n_q"] * (1 + case["paired"])
    length = (case["lo"] + case["hi"]) / 2
    wins = mates * max(1, math.ceil((length - case["k"] + 1) / stride))
    query = mates * (length + 8) + case["n_q"] * 16 + wins * s * 64
    if case["kind"] == "classify" and case["call"] == "shards":
        query = query * case["parts"] + case["n_q"] * 64 * (case["parts"] + 1)
    if case["kind"] in ("classify", "serve"):
        return {"bytes": query, "flops": 0}
    pairs = _n_bp(case) / stride * s
    build = _n_bp(case) + pairs * 4 + pairs / 4 * 8
    if case["kind"] == "build":
        return {"bytes": build + query, "flops": 0}
    return {"bytes": build + case["parts"] * query, "flops": 0}


def exact(case, seed):
    """Every output is a whole number that the integer arithmetic of the
    path gives exactly; there is none that is nearer."""
    return None

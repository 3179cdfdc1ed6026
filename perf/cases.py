"""The work that a user of this package has it do, as cases that can be timed.

A program that overlaps and aligns long reads packs a read set once, keeps the
packed store on the GPU, and then calls three things: ``dibella_candidate_pairs``
(which pairs share a retained k-mer), ``dibella_xdrop_batch`` and its host and
streaming forms (the seed-and-extend X-drop alignment of every pair, at one X),
and ``dibella_xdrop_traceback`` (the edits of the overlaps it accepted).  The
cases are those calls, from one seed record to a large batch.

Reads follow the shapes of the named workloads: a uniform-random genome (with
repeat families and tandem arrays in the repeat-rich one), reads from random
places and strands, errors split 20% substitution, 50% insertion and 30%
deletion, and seeds from the shared 17-mers whose multiplicity lies in the
workload's window.  Scoring is +1 / -1 / -1 everywhere, as in every named
workload.  All outputs are whole numbers (result records, seed records, edit
runs), so two implementations have to agree on every byte.
"""

import math

import numpy as np
import torch

import paper_2001_10049_gb300 as dib

# Read sets: genome bases, coverage, law of the read lengths, error rate range,
# multiplicity window, seeds per pair, repeat families, tandem bases.
READS = {
    # short reads of a small genome: the workload of a quick check
    "tiny": dict(genome=50_000, coverage=10.0, law="uniform", a=2000.0, b=6000.0, err=(0.15, 0.15), mult=8, seeds=1),
    # E. coli-sized: lognormal lengths of mean 9 kb, at 15% error
    "ecoli": dict(genome=4_600_000, coverage=30.0, law="lognormal", a=1000.0, b=60000.0, err=(0.15, 0.15), mult=8,
                  seeds=2),
    # uneven: lengths log-uniform from 500 b to 100 kb, error 5% to 35% by read
    "uneven": dict(genome=2_000_000, coverage=20.0, law="loguniform", a=500.0, b=100000.0, err=(0.05, 0.35), mult=8,
                   seeds=1),
    # repeat-rich: 10 families of two 5 kb copies at 3% divergence, 50 kb in tandem arrays
    "repeats": dict(genome=5_000_000, coverage=40.0, law="lognormal", a=1000.0, b=60000.0, err=(0.15, 0.15), mult=12,
                    seeds=1, families=10, tandem=50_000),
}
MATCH, MISMATCH, GAP = 1, -1, -1
K = 17


def listed():
    return [
        # One seed record, uploaded, aligned and read back: the smallest request
        # of a service, all latency.
        dict(name="one_seed_x25", do="align", reads="tiny", x=25, seeds=1, entry="host"),
        # The whole small workload at the smallest X: a batch too small to fill
        # the GPU.
        dict(name="tiny_batch_x7", do="align", reads="tiny", x=7, seeds=1000, entry="batch"),
        # A mid-sized request of a service (requests hold 1 to 4096 pairs).
        dict(name="request_200_x25", do="align", reads="ecoli", x=25, seeds=261, entry="batch"),
        # The largest request of a service at its largest X.
        dict(name="request_4096_x50", do="align", reads="ecoli", x=50, seeds=5395, entry="batch"),
        # E. coli-sized batches: a contiguous share of the candidate pairs, at
        # the X that ends chance pairs early and at the one that keeps them.
        dict(name="ecoli_x7", do="align", reads="ecoli", x=7, seeds=400_000, entry="batch"),
        dict(name="ecoli_x25", do="align", reads="ecoli", x=25, seeds=150_000, entry="batch"),
        # Lengths from 500 b to 100 kb at a large X: the widest bands and the
        # longest single extensions.
        dict(name="uneven_x50", do="align", reads="uneven", x=50, seeds=12_000, entry="batch"),
        # A repeat-rich genome's pairs streamed from pinned host memory in
        # chunks, two in flight.
        dict(name="repeats_stream_x15", do="align", reads="repeats", x=15, seeds=150_000, entry="stream"),
        # Candidate pairs of the small, the E. coli-sized and the repeat-rich
        # read set (the last one counted in hash passes, as for larger genomes).
        dict(name="candidates_tiny", do="candidates", reads="tiny", genome=50_000, coverage=10.0, parts=0),
        dict(name="candidates_ecoli", do="candidates", reads="ecoli", genome=4_600_000, coverage=30.0, parts=0),
        dict(name="candidates_repeats", do="candidates", reads="repeats", genome=5_000_000, coverage=40.0, parts=2),
        # The edits of accepted overlaps.
        dict(name="traceback_x25", do="traceback", reads="ecoli", x=25, seeds=2000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["align", "align", "align", "candidates", "traceback"])
    if do == "align":
        reads = rng.choice(["tiny", "ecoli", "uneven", "repeats"])
        x = rng.choice([7, 15, 25, 50, rng.randint(3, 55)])
        cap = 1000 if reads == "tiny" else int(min(400_000, 1.6e11 / _cells_per_seed(reads, x)))
        return dict(do="align", reads=reads, x=x, seeds=_log(rng, 1, cap),
                    entry=rng.choice(["host", "batch", "batch", "stream"]))
    if do == "candidates":
        reads = rng.choice(["tiny", "ecoli", "uneven", "repeats"])
        p = READS[reads]
        return dict(do="candidates", reads=reads, genome=_log(rng, 50_000, max(50_001, p["genome"])),
                    coverage=round(rng.uniform(10.0, p["coverage"] + 0.5), 1), parts=rng.choice([0, 0, 1, 3]))
    return dict(do="traceback", reads=rng.choice(["ecoli", "ecoli", "repeats"]), x=rng.choice([7, 15, 25, 35]),
                seeds=_log(rng, 20, 2000))


# ---- inputs ------------------------------------------------------------------

def _lengths(rng, p, genome, coverage):
    total, out = int(coverage * genome), []
    while total > 0:
        n = max(16, total // 4000)
        if p["law"] == "uniform":
            v = rng.uniform(p["a"], p["b"], n)
        elif p["law"] == "lognormal":  # mean 9 kb, sd 7 kb
            s2 = math.log(1.0 + (7000.0 / 9000.0) ** 2)
            v = rng.lognormal(math.log(9000.0) - s2 / 2, math.sqrt(s2), n)
        else:
            v = np.exp(rng.uniform(math.log(p["a"]), math.log(p["b"]), n))
        v = np.clip(v, p["a"], min(p["b"], genome)).astype(np.int64)
        keep = int(np.searchsorted(np.cumsum(v), total)) + 1
        out.append(v[:keep])
        total -= int(v[:keep].sum())
    return np.concatenate(out)


def _read_set(name, seed, genome=None, coverage=None):
    """(ASCII reads, offsets) of a read set, as a program that read a FASTA file has them."""
    p = READS[name]
    glen = p["genome"] if genome is None else genome
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def rand(n):
        return torch.rand(n, generator=gen, device="cuda")

    def bases(n):
        return torch.randint(0, 4, (n,), generator=gen, device="cuda", dtype=torch.uint8)

    g = bases(glen)
    for _ in range(p.get("families", 0)):
        unit = bases(5000)
        for _ in range(2):
            at = int(rng.integers(0, max(1, glen - 5000)))
            n = min(5000, glen - at)
            g[at:at + n] = torch.where(rand(n) < 0.03, bases(n), unit[:n])
    left = p.get("tandem", 0) * glen // p["genome"]
    while left > 0:
        n = min(int(rng.integers(500, 5001)), glen)
        at = int(rng.integers(0, glen - n + 1))
        unit = bases(int(rng.integers(2, 51)))
        g[at:at + n] = unit.repeat(n // len(unit) + 1)[:n]
        left -= n
    lens = _lengths(rng, p, glen, p["coverage"] if coverage is None else coverage)
    start = rng.integers(0, glen - lens + 1)
    back = rng.random(len(lens)) < 0.5
    err = rng.uniform(p["err"][0], p["err"][1] + 1e-12, len(lens))
    tl = torch.from_numpy(lens).cuda()
    off = torch.cumsum(tl, 0) - tl
    n = int(lens.sum())

    def per_base(v):
        return torch.repeat_interleave(torch.from_numpy(v).cuda(), tl, output_size=n)

    # base t of a forward read is genome[start + t], of a reverse one the complement of genome[start + len - 1 - t]
    fwd = ~per_base(back)
    idx = torch.arange(n, device="cuda") - torch.repeat_interleave(off, tl, output_size=n)
    idx = torch.where(fwd, per_base(start) + idx, per_base(start + lens - 1) - idx)
    b = g[idx]
    b = torch.where(fwd, b, 3 - b)
    del idx, fwd
    e = per_base(err.astype(np.float32))
    u = rand(n)
    gone = u < 0.3 * e
    sub = (u >= 0.3 * e) & (u < 0.5 * e)
    ins = (u >= 0.5 * e) & (u < e)
    del u, e
    b = torch.where(sub, (b + 1 + bases(n) % 3) & 3, b)
    cnt = 1 - gone.to(torch.int64) + ins.to(torch.int64)
    end = torch.cumsum(cnt, 0)
    out = bases(int(end[-1]))  # inserted bases stay as drawn
    at = end - cnt
    out[at[~gone]] = b[~gone]
    offs = torch.zeros(len(lens) + 1, dtype=torch.int64, device="cuda")
    offs[1:] = end[off + tl - 1]
    ascii = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")[out.long()]
    res = ascii.cpu().numpy(), offs.cpu().numpy()
    del b, gone, sub, ins, cnt, end, out, at, ascii
    torch.cuda.empty_cache()
    return res


def _store(name, seed, genome=None, coverage=None):
    return dib.ReadStore.from_ascii(*_read_set(name, seed, genome, coverage))


def _seeds(store, name, n, seed):
    """A contiguous run of n seed records of the read set's candidate pairs."""
    p = READS[name]
    recs, _ = store.candidate_pairs(k=K, mult_lo=2, mult_hi=p["mult"], max_seeds=p["seeds"])
    at = int(np.random.default_rng(seed + 1).integers(0, max(1, len(recs) - n + 1)))
    recs = recs[at:at + n].copy()
    torch.cuda.empty_cache()
    return recs


def _pinned(a, width):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1, width).copy()).pin_memory()


def prepare(case, seed):
    if case["do"] == "candidates":
        return _prepare_candidates(case, seed)
    store = _store(case["reads"], seed)
    if case["do"] == "traceback":
        return _prepare_traceback(case, seed, store)
    pairs = _seeds(store, case["reads"], case["seeds"], seed)
    n = len(pairs)
    s = dict(case=case, store=store, n=n, scoring=dib.Scoring(MATCH, MISMATCH, GAP, case["x"]))
    if case["entry"] == "stream":
        chunk = max(1, min(n, 65536))
        s.update(host_pairs=_pinned(pairs, 24), host_results=torch.zeros((n, 40), dtype=torch.uint8).pin_memory(),
                 chunk=chunk, ws_bytes=dib.dibella_xdrop_workspace_bytes(chunk, max(store.max_len, 1)),
                 streams=[torch.cuda.Stream(), torch.cuda.Stream()])
        s["staging"] = [torch.empty(dib.dibella_staging_bytes(chunk), dtype=torch.uint8, device="cuda")
                        for _ in range(2)]
        s["workspace"] = [torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda") for _ in range(2)]
        return s
    s["aligner"] = dib.Aligner(store, n, k=K)
    s["pairs"] = pairs
    s["aligner"].upload_pairs(pairs)
    return s


def _prepare_candidates(case, seed):
    store = _store(case["reads"], seed, case["genome"], case["coverage"])
    p = READS[case["reads"]]
    s = dict(case=case, store=store, mult=p["mult"], seeds=p["seeds"])
    # room for the seed records: about as much as the package's own ReadStore.candidate_pairs takes
    cap = 4096 + int(case["genome"] * case["coverage"]) // 16
    s["cap"] = cap
    s["out"] = torch.zeros((cap, 24), dtype=torch.uint8, device="cuda")
    s["counts"] = torch.zeros(7, dtype=torch.int64, device="cuda")
    if case["parts"]:
        s["occ"] = max(4096, store.n_bases // 4)
        ws = dib.dibella_candidate_workspace_bytes_parts(store.n_reads, store.n_bases, store.max_len, K,
                                                         case["parts"], s["occ"])
    else:
        ws = dib.dibella_candidate_workspace_bytes(store.n_reads, store.n_bases, K, p["mult"])
    s["ws"] = torch.empty(ws, dtype=torch.uint8, device="cuda")
    s["ws_bytes"] = ws
    return s


def _prepare_traceback(case, seed, store):
    """Seeds of accepted overlaps: the best of their pair, 2 kb or more of A at 0.2 per column or better."""
    n = case["seeds"]
    pairs = _seeds(store, case["reads"], 16 * n, seed)
    res = dib.Aligner(store, len(pairs), k=K).align(pairs, dib.Scoring(MATCH, MISMATCH, GAP, case["x"]))
    span = res["end_a"].astype(np.int64) - res["begin_a"]
    ok = ((res["status"] & dib.RES_BEST_OF_PAIR) != 0) & (span >= 2000) & (res["score"] >= 0.2 * span)
    acc = np.ascontiguousarray(pairs[ok][:n])
    n = len(acc)
    lanes = max(1, min(n, 24 * torch.cuda.get_device_properties("cuda").multi_processor_count))
    moves = 1 << 20
    ws = dib.dibella_traceback_workspace_bytes(lanes, store.max_len, moves)
    return dict(case=case, store=store, n=n, scoring=dib.Scoring(MATCH, MISMATCH, GAP, case["x"]),
                pairs=torch.from_numpy(acc.view(np.uint8).reshape(n, 24).copy()).cuda(),
                results=torch.zeros((n, 40), dtype=torch.uint8, device="cuda"),
                ops=torch.zeros((n, 8192), dtype=torch.int32, device="cuda"),
                n_ops=torch.zeros(n, dtype=torch.int32, device="cuda"), lanes=lanes, moves=moves,
                ws=torch.empty(ws, dtype=torch.uint8, device="cuda"), ws_bytes=ws)


# ---- one pass ----------------------------------------------------------------

def run(s):
    case, st = s["case"], s["store"]
    if case["do"] == "candidates":
        if case["parts"]:
            dib.dibella_candidate_pairs_parts(st.words, st.word_offsets, st.lengths, st.n_reads, st.n_bases, st.max_len,
                                              K, 2, s["mult"], s["seeds"], 0, case["parts"], s["occ"], s["out"],
                                              s["cap"], s["counts"], s["ws"], s["ws_bytes"])
        else:
            dib.dibella_candidate_pairs(st.words, st.word_offsets, st.lengths, st.n_reads, st.n_bases, st.max_len, K,
                                        2, s["mult"], s["seeds"], 0, s["out"], s["cap"], s["counts"], s["ws"],
                                        s["ws_bytes"])
        return s["out"], s["counts"]
    if case["do"] == "traceback":
        dib.dibella_xdrop_traceback(st.words, st.word_offsets, st.lengths, st.n_reads, st.max_len, s["pairs"], s["n"],
                                    K, s["scoring"], s["results"], s["ops"], 8192, s["n_ops"], s["lanes"], s["moves"],
                                    s["ws"], s["ws_bytes"])
        return s["results"], s["ops"], s["n_ops"]
    if case["entry"] == "host":
        res = s["aligner"].align(s["pairs"], s["scoring"])
        return res.view(np.uint8).reshape(-1, 40)
    if case["entry"] == "stream":
        dib.dibella_xdrop_stream(st.words, st.word_offsets, st.lengths, st.n_reads, s["host_pairs"], s["n"],
                                 s["chunk"], K, s["scoring"], s["host_results"], s["staging"], s["workspace"],
                                 s["ws_bytes"], s["streams"])
        return s["host_results"]
    s["aligner"].run(s["n"], s["scoring"])
    return s["aligner"].results[:s["n"]]


# ---- what a pass cannot do without ----------------------------------------------

def _mean_pair_bases(reads):
    """Bases of both reads of a mean candidate pair (long reads are in more pairs)."""
    return {"tiny": 9e3, "ecoli": 28e3, "uneven": 80e3, "repeats": 28e3}[reads]


def _cells_per_seed(reads, x):
    """Cells that the X-drop rule evaluates for a mean seed record: a true
    overlap keeps a band of about 1.1 x cells over the shared span, and from X
    of about 10 on a chance pair (a share of the candidates that the read set's
    size fixes) one of about 5.3 x to the end of the shorter read."""
    chance = {"tiny": 0.02, "ecoli": 0.5, "uneven": 0.65, "repeats": 0.65}[reads]
    bases = _mean_pair_bases(reads)
    true = (1.0 - chance) * 0.4 * bases * 1.1 * x
    return true + (chance * 0.6 * bases * 5.3 * x if x > 10 else chance * 2000.0)


def work(case):
    p = READS[case["reads"]]
    if case["do"] == "candidates":
        bases = case["genome"] * case["coverage"]
        # every base read once at 2 bits, every seed record written (about one for 80 bases)
        return {"bytes": bases / 4 + 24 * bases / 80, "flops": 0.0}
    n = case["seeds"] if case["reads"] != "tiny" else min(case["seeds"], 1200)
    seq = min(n * _mean_pair_bases(case["reads"]), p["genome"] * p["coverage"] * 2)
    cells = n * _cells_per_seed(case["reads"], case["x"])
    if case["do"] == "traceback":  # true overlaps only
        cells = n * 0.4 * _mean_pair_bases(case["reads"]) * 1.1 * case["x"]
    # both reads of each pair at 2 bits (the store at most once), the seed record in, the result record out;
    # 8 integer operations to a cell
    extra = n * 8 * 1000.0 if case["do"] == "traceback" else 0.0  # about a thousand runs of edits, read and written
    return {"bytes": seq / 4 + 64 * n + extra, "flops": 8.0 * cells}


def exact(case, seed):
    """Nothing: every output is whole numbers, which have to be equal as they are."""
    return None

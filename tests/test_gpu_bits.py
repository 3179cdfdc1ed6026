"""The bit-sliced form on the GPU (default schedule, unit scores, X from 1 to 59):
at the edges of its score planes and of the rule that chooses it, and on a batch
whose extensions crowd the warps and the pool of suspended extensions.  Whole
numbers: nothing may differ."""

import random

import numpy as np
import pytest

import workloads
from gpu_util import WIDE_ALL, assert_same, gpu_align, make_pairs, oracle_align, rc, reads_to_arrays, schedule

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def c1():
    return workloads.generate("c1_tiny")


@pytest.mark.parametrize("X", [1, 11, 12, 27, 28, 59, 60])
def test_plane_edges(c1, X):
    """4 planes to X = 11, 5 to 27, 6 to 59, the int16 forms above."""
    pairs = c1.pairs[:250]
    sc = (1, -1, -1, X)
    assert_same(gpu_align(c1.reads, c1.offsets, pairs, 17, sc), oracle_align(c1.reads, c1.offsets, pairs, 17, sc),
                "X=%d" % X)


@pytest.mark.parametrize("X", [9, 25, 50])
def test_crowded_warps(X):
    """60,000 seeds at random places of short reads: unrelated, related,
    low-complexity and tiny ones, so that bands widen and end all the time and
    the pool (sized by the longest read) runs out; against the int16 form on
    every record and the oracle on a sample."""
    rng = random.Random(X)
    rand = lambda n: "".join(rng.choice("ACGT") for _ in range(n))
    genome = rand(900)
    reads = [genome[s:s + rng.randint(200, 600)] for s in (0, 50, 120, 300)]
    reads += [rand(rng.randint(100, 700)) for _ in range(20)] + [rand(3) * 150, rand(2) * 200, "A" * 400, "AC", "A"]
    reads += [rc(r) for r in reads[:6]]
    recs = []
    for _ in range(60000):
        a, b = rng.randrange(len(reads)), rng.randrange(len(reads))
        recs.append((a, b, rng.randrange(len(reads[a])), rng.randrange(len(reads[b])), rng.randint(0, 1)))
    ascii, offs = reads_to_arrays(reads)
    pairs = make_pairs(recs)
    sc = (1, -1, -1, X)
    got = gpu_align(ascii, offs, pairs, 1, sc)
    assert_same(got, gpu_align(ascii, offs, pairs, 1, sc, sched=schedule(**WIDE_ALL)), "int16 form, X=%d" % X)
    idx = np.sort(np.random.default_rng(X).choice(len(pairs), 500, replace=False))
    exp = oracle_align(ascii, offs, pairs[idx], 1, sc)
    sub = got[idx].copy()
    for r in (sub, exp):
        r["status"] &= ~4  # the best-of-pair flag depends on the neighbouring records
    assert_same(sub, exp, "oracle, X=%d" % X)


@pytest.mark.parametrize("moves_words,ops_per_seed", [(1 << 18, 4096), (30000, 4096), (2500, 4096), (300, 64), (1 << 18, 7)])
@pytest.mark.parametrize("X", [5, 25, 59])
def test_traceback_equals_general_form(X, moves_words, ops_per_seed):
    """Scores and X doubled give the same alignments, but by the general form:
    every run, run count and status (moves or runs that do not fit among them)
    is the same, and the scores are doubled.  The capacities take the two
    extensions together, one after the other, and beyond what fits."""
    import torch
    import paper_2001_10049_gb300 as dib
    rng = random.Random(X + moves_words)
    rand = lambda n: "".join(rng.choice("ACGT") for _ in range(n))

    def noisy(s, e):
        out = []
        for ch in s:
            r = rng.random()
            out.append("" if r < 0.3 * e else (rng.choice("ACGT") if r < 0.5 * e else ch + (rng.choice("ACGT") if r < e else "")))
        return "".join(out)

    core = rand(2500)
    reads = [noisy(core, 0.15) for _ in range(6)] + [core, core, rand(1800), rand(2000), rand(4) * 300, "A" * 500, rand(40)]
    reads += [rc(r) for r in reads[:3]]
    recs = [(a, b, p, min(p, len(reads[b]) - 31), st) for a in range(len(reads)) for b in range(len(reads))
            for st in (0, 1) for p in (0, len(reads[a]) // 2, max(0, len(reads[a]) - 31))]
    recs = [r for r in recs if r[3] >= 0]
    ascii, offs = reads_to_arrays(reads)
    al = dib.Aligner(dib.ReadStore.from_ascii(ascii, offs), len(recs), k=31)
    pairs = make_pairs(recs)
    res, ops, n_ops = al.traceback(pairs, (1, -1, -1, X), ops_per_seed=ops_per_seed, moves_words=moves_words)
    res2, ops2, n_ops2 = al.traceback(pairs, (2, -2, -2, 2 * X), ops_per_seed=ops_per_seed, moves_words=moves_words)
    assert np.array_equal(n_ops, n_ops2) and np.array_equal(ops, ops2)
    for f in ("begin_a", "end_a", "begin_b", "end_b", "status", "cells"):
        assert np.array_equal(res[f], res2[f]), f
    for f in ("score", "score_left", "score_right"):
        assert np.array_equal(2 * res[f], res2[f]), f
    torch.cuda.synchronize()

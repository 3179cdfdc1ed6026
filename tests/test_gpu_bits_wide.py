"""Wide bands of the bit-sliced form on the GPU (default schedule, unit scores):
poly-A against (AC)n, whose band is a quarter of the length at its widest, so that
6, 12, 20 and 36 kb go to 2 and 4 words a lane, the CTA form and the global form;
with a roomy pool of suspended extensions and with one that is full.  Records
against the oracle.  The traceback of wide and of drifting bands against its
general form.  Whole numbers: nothing may differ."""

import random

import numpy as np
import pytest

import workloads  # noqa: F401  (builds its library before the first GPU call)
from gpu_util import assert_same, make_pairs, oracle_align, rc, reads_to_arrays

pytestmark = pytest.mark.gpu


def wide_reads(longest):
    """(AC)n and poly-A reads in turn; read 2 i and 2 i + 1 have the same length."""
    out = []
    for n in (6000, 12000, 20000, 36000):
        if n <= longest:
            out += ["AC" * (n // 2), "A" * n]
    return out


@pytest.mark.parametrize("room", ["pool", "full"])
@pytest.mark.parametrize("X", [7, 25, 59])
def test_wide_bands(X, room):
    import paper_2001_10049_gb300 as dib
    rng = random.Random(X)
    rand = lambda n: "".join(rng.choice("ACGT") for _ in range(n))
    wide = wide_reads(36000 if room == "pool" else 20000)
    genome = rand(1500)
    reads = wide + [genome[s:s + rng.randint(300, 900)] for s in (0, 90, 300, 500)] + [rand(900) for _ in range(16)]
    reads += ["C" + wide[1], wide[0] + rand(700)]
    recs = [(2 * i, 2 * i + 1, p, p, 0) for i in range(len(wide) // 2) for p in (0, 1)]
    recs += [(1, 0, 5990, 5990, 1), (len(reads) - 2, 0, 0, 0, 0), (len(reads) - 1, 1, 2, 2, 0)]
    if room == "full":  # (a dozen wide pairs, and as many seeds as crowd the pool)
        recs += [(2 * (i % 2), 2 * (i % 2) + 1, i, i, 0) for i in range(12)]
    for _ in range(500):
        a, b = rng.randrange(len(wide), len(reads) - 2), rng.randrange(len(wide), len(reads) - 2)
        recs.append((a, b, rng.randrange(len(reads[a])), rng.randrange(len(reads[b])), rng.randint(0, 1)))
    ascii, offs = reads_to_arrays(reads)
    pairs = make_pairs(recs)
    al = dib.Aligner(dib.ReadStore.from_ascii(ascii, offs), len(pairs), k=1)
    if room == "full":  # the smallest band in the workspace, and the pool with it
        al.workspace_bytes = dib.dibella_xdrop_workspace_bytes(len(pairs), 1)
    got = al.align(pairs, (1, -1, -1, X))
    counters = dib.dibella_batch_counters(al.workspace)
    assert_same(got, oracle_align(ascii, offs, pairs, 1, (1, -1, -1, X)), "X=%d, %s" % (X, room))
    assert counters["cells_ladder"] > 0 and counters["cells_smem"] > 0  # the 4-word launch and the CTA form
    if room == "pool":
        assert counters["cells_global"] > 0
    else:
        assert counters["cells_restarted"] > 0
    assert 0 < counters["escalated_narrow"] <= 17 * 2 * len(pairs)


@pytest.mark.parametrize("X", [7, 25, 59])
def test_traceback_of_wide_and_drifting_bands(X):
    """Scores and X doubled: the general form (see test_gpu_bits).  Bands beyond the
    512- and 1,024-cell windows, and bands that leave the middle by 1,500 cells to
    either side (every eighth base deleted)."""
    import torch
    import paper_2001_10049_gb300 as dib
    rng = random.Random(X)
    core = "".join(rng.choice("ACGT") for _ in range(12000))
    thin = "".join(ch for q, ch in enumerate(core) if q % 8)
    reads = wide_reads(6000) + ["AC" * 1500, "A" * 3000, core, thin, rc(core)]
    recs = [(0, 1, 0, 0, 0), (1, 0, 5968, 5968, 0), (2, 3, 0, 0, 0), (3, 2, 1500, 1500, 1), (4, 5, 0, 0, 0),
            (5, 4, 0, 0, 0), (4, 5, 6000, 5250, 0), (5, 4, 5250, 6000, 0), (6, 5, 6000, 5250, 1), (4, 5, 11968, 10468, 0)]
    ascii, offs = reads_to_arrays(reads)
    al = dib.Aligner(dib.ReadStore.from_ascii(ascii, offs), len(recs), k=31)
    pairs = make_pairs(recs)
    res, ops, n_ops = al.traceback(pairs, (1, -1, -1, X), ops_per_seed=16384, moves_words=1 << 22)
    res2, ops2, n_ops2 = al.traceback(pairs, (2, -2, -2, 2 * X), ops_per_seed=16384, moves_words=1 << 22)
    assert np.array_equal(n_ops, n_ops2) and np.array_equal(ops, ops2) and (n_ops > 0).all()
    for f in ("begin_a", "end_a", "begin_b", "end_b", "status", "cells"):
        assert np.array_equal(res[f], res2[f]), f
    for f in ("score", "score_left", "score_right"):
        assert np.array_equal(2 * res[f], res2[f]), f
    if X > 7:  # the drifting overlap is followed to its end
        assert res["end_a"][4] > 11000
    torch.cuda.synchronize()

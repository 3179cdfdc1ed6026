"""The bucket count of dibella_candidate_pairs at the sizes where it can go
wrong, against the oracle: buckets of more codes than the hash table takes,
frequent codes, buckets whose retained occurrences leave shared memory, codes of
64-bit tags, one bucket, many buckets.  Byte-identical records, equal counts."""

import random

import numpy as np
import pytest

from oracle import candidates as oc

pytestmark = pytest.mark.gpu


def arrays(reads):
    ascii = np.frombuffer("".join(reads).encode(), dtype=np.uint8)
    return ascii, np.cumsum([0] + [len(r) for r in reads]).astype(np.int64)


def check(reads, k, lo, hi, max_seeds=1000, gap=0, n_parts=0):
    import paper_2001_10049_gb300 as dib
    ascii, offs = arrays(reads)
    store = dib.ReadStore.from_ascii(ascii, offs)
    if n_parts:
        got, st = store.candidate_pairs_parts(k=k, mult_lo=lo, mult_hi=hi, max_seeds=max_seeds, min_seed_gap=gap,
                                              n_parts=n_parts)
    else:
        got, st = store.candidate_pairs(k=k, mult_lo=lo, mult_hi=hi, max_seeds=max_seeds, min_seed_gap=gap)
    exp, est = oc.candidate_pairs(ascii, offs, k, lo, hi, max_seeds, gap)
    assert st["status"] == 0
    for key in ("instances", "retained_kmers", "candidate_pairs", "occurrence_pairs"):
        assert st[key] == est[key], key
    assert got.tobytes() == exp.view(got.dtype).tobytes()


def same_bucket_kmers(n, k, bits, seed):
    """n distinct k-mers whose mixed canonical codes share their highest bits."""
    rng = np.random.default_rng(seed)
    mask = (1 << (2 * k)) - 1
    out = {}
    while len(out) < n:
        b = rng.integers(0, 4, (200000, k))
        w = (4 ** np.arange(k - 1, -1, -1, dtype=np.uint64))
        fw = (b.astype(np.uint64) * w).sum(1)
        rc = ((3 - b[:, ::-1]).astype(np.uint64) * w).sum(1)
        c = np.minimum(fw, rc)
        top = ((c * np.uint64(0x9E3779B97F4A7C15)) & np.uint64(mask)) >> np.uint64(2 * k - bits)
        for i in np.flatnonzero(top == 1):
            out[int(c[i])] = b[i]
    return ["".join("ACGT"[x] for x in v) for v in list(out.values())[:n]]


@pytest.mark.parametrize("n_parts", [0, 1])
def test_more_codes_than_the_table(n_parts):
    kmers = same_bucket_kmers(5500, 17, 8, 1)
    check(kmers + kmers[:3000] + kmers[1000:1500], 17, 2, 8, n_parts=n_parts)


@pytest.mark.parametrize("k", [13, 17, 23])
def test_frequent_and_retained_codes(k):
    rng = random.Random(k)
    rand = lambda n: "".join(rng.choice("ACGT") for _ in range(n))
    core = rand(1500)
    reads = [core[s:s + 400] for s in range(0, 1100, 50)] * 2  # every occurrence retained
    reads += ["A" * 3000, rand(2) * 2000, rand(7) * 500]        # far above the window
    reads += [rand(300) for _ in range(40)]
    rng.shuffle(reads)
    check(reads, k, 2, 32)
    check(reads, k, 2, 8, max_seeds=2, gap=30, n_parts=2)


@pytest.mark.parametrize("n_bases", [40, 2000, 2100, 70000, 5_000_000])
def test_bucket_counts(n_bases):
    rng = random.Random(n_bases)
    genome = np.random.default_rng(n_bases).integers(0, 4, max(30, n_bases // 6))
    text = "".join("ACGT"[b] for b in genome)
    reads = []
    while sum(map(len, reads)) < n_bases:
        n = rng.randint(1, min(len(text), 3000))
        s = rng.randint(0, len(text) - n)
        reads.append(text[s:s + n])
    check(reads, 17, 2, 12, max_seeds=2)

"""dibella_candidate_pairs on buckets that are thinned before they are counted
(more than 16,384 occurrences in one): codes of many thousand occurrences, and in
the same buckets codes at both edges of the window spread over the whole input.
Against the oracle: byte-identical records, equal counts."""

import random

import numpy as np
import pytest

from test_gpu_candidates_buckets import check

pytestmark = pytest.mark.gpu


def first_bucket_kmers(n, k, bits, seed):
    """n distinct k-mers whose mixed canonical codes begin with `bits` zeros: the bucket of poly-A."""
    rng = np.random.default_rng(seed)
    mask = np.uint64((1 << (2 * k)) - 1)
    w = (4 ** np.arange(k - 1, -1, -1, dtype=np.uint64))
    out = {}
    while len(out) < n:
        b = rng.integers(0, 4, (200000, k))
        fw = (b.astype(np.uint64) * w).sum(1)
        rc = ((3 - b[:, ::-1]).astype(np.uint64) * w).sum(1)
        c = np.minimum(fw, rc)
        top = ((c * np.uint64(0x9E3779B97F4A7C15)) & mask) >> np.uint64(2 * k - bits)
        for i in np.flatnonzero(top == 0):
            out[int(c[i])] = "".join("ACGT"[x] for x in b[i])
    return list(out.values())[:n]


@pytest.mark.parametrize("k,hi", [(13, 8), (17, 2), (17, 8), (17, 32), (23, 8)])
@pytest.mark.parametrize("n_parts", [0, 2])
def test_big_buckets(k, hi, n_parts):
    rng = random.Random(k + hi)
    rand = lambda n: "".join(rng.choice("ACGT") for _ in range(n))
    kmers = first_bucket_kmers(120, k, 7, k)
    reads = ["A" * (k - 1 + n) for n in (9000, 40000, 1, 3)]       # one code, 49,004 times
    reads += [rand(2) * 6000, rand(5) * 4000, rand(44) * 900]      # several frequent codes
    for q, m in enumerate(kmers):                                  # 1, hi or hi + 1 occurrences of each
        reads += [m] * (1, hi, hi + 1)[q % 3]
    reads += [rand(600) for _ in range(60)] + [rand(300)] * 2
    rng.shuffle(reads)
    check(reads, k, min(2, hi), hi, n_parts=n_parts)


def test_one_bucket_holds_everything():
    """k = 3: at most 32 codes, every one of them frequent; then the last code's count is exactly the window's."""
    rng = random.Random(3)
    text = "".join(rng.choice("ACGT") for _ in range(60000))
    check([text[i:i + 900] for i in range(0, 60000, 900)], 3, 2, 32)
    check(["A" * 30000] + ["CCC"] * 32, 3, 2, 32)


def test_one_code_is_not_one_blocks_work():
    """20 Mb of poly-A take no longer than a few times 20 Mb of random bases
    (42 ms against 1.4 when one block counted them alone)."""
    import torch
    import paper_2001_10049_gb300 as dib
    rng = np.random.default_rng(5)
    best = {}
    for name in ("random", "poly-A"):
        reads = 2000
        flat = np.full(reads * 10000, 65, np.uint8)
        if name == "random":
            flat = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, reads * 10000)]
        st = dib.ReadStore.from_ascii(flat, np.arange(reads + 1, dtype=np.int64) * 10000)
        nb = st.n_bases
        wsb = dib.dibella_candidate_workspace_bytes(st.n_reads, nb, 17, 8)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        out = torch.empty((1 << 20, 24), dtype=torch.uint8, device="cuda")
        counts = torch.zeros(7, dtype=torch.int64, device="cuda")
        ms = []
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            dib.dibella_candidate_pairs(st.words, st.word_offsets, st.lengths, st.n_reads, nb, st.max_len, 17, 2, 8, 1, 0,
                                        out, len(out), counts, ws, wsb)
            e1.record()
            torch.cuda.synchronize()
            ms.append(e0.elapsed_time(e1))
        assert int(counts[2]) == reads * (10000 - 16) and int(counts[5]) == 0
        best[name] = min(ms)
    assert best["poly-A"] <= 4 * best["random"], best

"""dibella_candidate_pairs_parts where a pass is numbered by three bucket digits
(more than 201 M occurrences expected: stated so here, the input is small), and
buckets of several times the codes that the table takes.  Against the oracle."""

import random

import numpy as np
import pytest

from oracle import candidates as oc
from test_gpu_candidates_buckets import arrays, check, same_bucket_kmers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bases", [3072 << 16, (3072 << 16) + 65536, 1 << 28])
def test_bucket_digits(n_bases):
    import torch
    import paper_2001_10049_gb300 as dib
    rng = random.Random(11)
    genome = "".join(rng.choice("ACGT") for _ in range(20000))
    reads = []
    for _ in range(60):
        n, s = rng.randint(1, 3000), rng.randint(0, 17000)
        reads.append(genome[s:s + n])
    reads += ["A" * 25000, "AC" * 300]
    ascii, offs = arrays(reads)
    st = dib.ReadStore.from_ascii(ascii, offs)
    occ = 1 << 20
    wsb = dib.dibella_candidate_workspace_bytes_parts(st.n_reads, n_bases, st.max_len, 17, 1, occ)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    out = torch.zeros((occ, 24), dtype=torch.uint8, device="cuda")
    counts = torch.zeros(7, dtype=torch.int64, device="cuda")
    dib.dibella_candidate_pairs_parts(st.words, st.word_offsets, st.lengths, st.n_reads, n_bases, st.max_len, 17, 2, 12, 2,
                                      0, 1, occ, out, occ, counts, ws, wsb)
    c = counts.cpu().numpy()
    exp, est = oc.candidate_pairs(ascii, offs, 17, 2, 12, 2, 0)
    assert c[5] == 0 and c[2] == est["instances"] and c[3] == est["retained_kmers"] and c[4] == est["occurrence_pairs"]
    assert len(exp) > 500 and out[:c[0]].cpu().numpy().tobytes() == exp.tobytes()


def test_many_codes_in_one_bucket():
    kmers = same_bucket_kmers(15000, 17, 8, 2)
    check(kmers + kmers[:9000] + kmers[4000:4500], 17, 2, 8)


def test_one_large_pass_against_four():
    """515 M random bases: in one pass the buckets would hold several times the
    codes that the table takes if they were numbered by two digits (81 ms then; 33
    with three, 36 in four passes, and half as much again is allowed)."""
    import torch
    import paper_2001_10049_gb300 as dib
    rng = np.random.default_rng(6)
    n_reads, n = 51500, 10000
    flat = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n_reads * n, dtype=np.uint8)]
    st = dib.ReadStore.from_ascii(flat, np.arange(n_reads + 1, dtype=np.int64) * n)
    del flat
    occ = 1 << 26
    ms, recs = {}, {}
    for parts in (1, 4):
        wsb = dib.dibella_candidate_workspace_bytes_parts(st.n_reads, st.n_bases, st.max_len, 17, parts, occ)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        out = torch.empty((occ, 24), dtype=torch.uint8, device="cuda")
        counts = torch.zeros(7, dtype=torch.int64, device="cuda")
        t = []
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            dib.dibella_candidate_pairs_parts(st.words, st.word_offsets, st.lengths, st.n_reads, st.n_bases, st.max_len, 17,
                                              2, 8, 1, 0, parts, occ, out, occ, counts, ws, wsb)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        ms[parts] = min(t)
        c = counts.cpu().numpy()
        assert c[5] == 0 and c[2] == n_reads * (n - 16) and c[0] > 1_000_000
        recs[parts] = out[:c[0]].clone()
        del ws, out
    assert torch.equal(recs[1], recs[4])
    assert ms[1] <= 1.5 * ms[4], ms

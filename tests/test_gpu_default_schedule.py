"""The built-in schedule passed explicitly is the same as none: the bit-sliced form
where it applies (a batch of 9 launches, more in the other forms), so that what
dibella_get_default_schedule and dibella_autotune return is as fast as no schedule.
Every other schedule, and the built-in one elsewhere, is followed as given."""

import pytest

import workloads
from gpu_util import assert_same, oracle_align, schedule

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def batch():
    import paper_2001_10049_gb300 as dib
    c1 = workloads.generate("c1_tiny")
    return c1, dib.Aligner(dib.ReadStore.from_ascii(c1.reads, c1.offsets), len(c1.pairs), k=17)


def align(batch, scoring, sched):
    """The records, and whether the batch ran in the bit-sliced form."""
    import paper_2001_10049_gb300 as dib
    c1, al = batch
    res = al.align(c1.pairs, dib.Scoring(*scoring), sched=sched)
    return res, dib.dibella_last_launch_count() == 9


@pytest.mark.parametrize("scoring,applies", [((1, -1, -1, 1), True), ((1, -1, -1, 25), True), ((1, -1, -1, 59), True),
                                             ((1, -1, -1, 0), False), ((1, -1, -1, 60), False), ((2, -1, -1, 25), False)])
def test_built_in_schedule(batch, scoring, applies):
    import paper_2001_10049_gb300 as dib
    c1 = batch[0]
    exp = oracle_align(c1.reads, c1.offsets, c1.pairs, 17, scoring)
    for sched, bits in ((None, applies), (dib.dibella_get_default_schedule(), applies),
                        (schedule(narrow_unroll=16), False)):
        res, took = align(batch, scoring, sched)
        assert took == bits
        assert_same(res, exp, str(scoring))


def test_own_default(batch):
    """A default that the caller set is not the built-in schedule; the built-in one passed to the call is."""
    import paper_2001_10049_gb300 as dib
    built_in = dib.dibella_get_default_schedule()
    sc = (1, -1, -1, 25)
    try:
        dib.dibella_set_default_schedule(schedule(narrow_unroll=16))
        assert not align(batch, sc, None)[1]
        assert not align(batch, sc, dib.dibella_get_default_schedule())[1]
        assert align(batch, sc, built_in)[1]
    finally:
        dib.dibella_set_default_schedule(built_in)
    assert align(batch, sc, None)[1]


def test_autotune_returns_the_fastest(batch):
    """The tiny batch takes about five times as long in the int16 forms."""
    import paper_2001_10049_gb300 as dib
    c1, al = batch
    al.upload_pairs(c1.pairs)
    st = al.store
    best, ms, tried = dib.dibella_autotune(st.words, st.word_offsets, st.lengths, st.n_reads, al.pairs, len(c1.pairs), 17,
                                           dib.Scoring(1, -1, -1, 7), al.results, al.workspace, al.workspace_bytes,
                                           repeats=1)
    assert best.as_dict() == dib.dibella_get_default_schedule().as_dict() and tried >= 10 and ms > 0

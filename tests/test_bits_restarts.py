"""The bit-sliced form with a pool of suspended extensions that has no room (its
kernel source on the CPU, as in test_bits_emulation): how often an extension
starts over is bounded by the forms it goes through, not by the queue's slots."""

import ctypes
import random

import numpy as np
import pytest

import oracle
import paper_2001_10049_gb300 as dib
from test_bits_emulation import compile_emulation, sequences


@pytest.fixture(scope="module")
def emulations(tmp_path_factory):
    folder = tmp_path_factory.mktemp("restarts")
    return {lanes: compile_emulation(folder, lanes) for lanes in (32, 2)}


def emulate(emu, pairs, nb, X, reserve, young, pool, slots):
    reads = [s for p in pairs for s in p]
    ascii = np.frombuffer("".join(reads).encode(), dtype=np.uint8)
    offs = np.cumsum([0] + [len(r) for r in reads]).astype(np.int64)
    words, woffs, lens = dib.dibella_pack_reads(ascii, offs)
    n = len(pairs)
    copy = (((lens.astype(np.int64) + 15) // 16) + 3) // 4 * 4
    a0 = np.ascontiguousarray(woffs[0::2] * 16)
    b0 = np.ascontiguousarray((woffs[1::2] + copy[1::2]) * 16 + lens[1::2] - 1)
    la, lb = np.ascontiguousarray(lens[0::2]), np.ascontiguousarray(lens[1::2])
    out = np.zeros((n, 4), dtype=np.int64)
    stats = np.zeros(4, dtype=np.int64)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    rc = emu.bits_emulate(nb, p(words), ctypes.c_longlong(len(words)), p(a0), p(b0), p(la), p(lb), n, X, reserve, young,
                          16, pool, slots, p(out), p(stats))
    assert rc == 0
    for i, (a, b) in enumerate(pairs):
        assert tuple(out[i]) == oracle.extend(a, b, 1, -1, -1, X)[:4], (i, a[:40], b[:40])
    return stats


@pytest.mark.parametrize("pool", [0, 1 << 20])
def test_band_beyond_a_warp(emulations, pool):
    """A band of up to 1,500 cells: it outgrows 32 lanes, and was narrow when it began."""
    stats = emulate(emulations[32], [("AC" * 3000, "A" * 6000)], 5, 25, 5, 500, pool, 100)
    assert stats[3] <= 3


@pytest.mark.parametrize("X", [13, 27])
@pytest.mark.parametrize("pool", [0, 700])
def test_crowded_warp(emulations, X, pool):
    """At most 2 lanes to an extension: 36 pairs crowd a warp and outgrow their
    lanes.  Each may start over 16 times there and then goes on to the whole-warp
    launch."""
    pairs = sequences(random.Random(8), 36, 300)
    for reserve, young in ((4, 100), (2, 0)):
        stats = emulate(emulations[2], pairs, 5, X, reserve, young, pool, 1000)
        assert stats[3] <= 17 * len(pairs)

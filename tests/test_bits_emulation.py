"""The bit-sliced X-drop form, its kernel source run lane by lane on the CPU
(tests/bits_emulation.cpp), against the oracle: best score, its cell and the
evaluated-cell count of every extension, for groups of 1 to 32 lanes.

Whole numbers: nothing may differ."""

import ctypes
import os
import random
import subprocess

import numpy as np
import pytest

import oracle
import paper_2001_10049_gb300 as dib

HERE = os.path.dirname(os.path.abspath(__file__))
# form, planes, lanes reserved, antidiagonals reserved for, extensions per warp, pool words, queue slots,
# most lanes of an extension: roomy and tight packing, a pool and a queue that run out, one extension
# per warp, bands that need a whole warp (also without a pool), and the whole-warp form alone
CASES = [(4, 4, 2, 50, 16, 1 << 20, 1000, 32), (5, 5, 6, 200, 16, 1 << 20, 1000, 32),
         (5, 5, 2, 0, 16, 1 << 20, 1000, 32), (5, 5, 2, 0, 16, 700, 1000, 32), (5, 5, 2, 0, 16, 1 << 20, 5, 32),
         (5, 5, 16, 1000, 1, 1 << 20, 1000, 32), (6, 6, 10, 400, 5, 1 << 20, 1000, 32),
         (5, 5, 4, 100, 16, 1 << 20, 1000, 2), (5, 5, 4, 100, 16, 0, 1000, 2), (6, 6, 2, 100, 16, 1 << 20, 1000, 2),
         (54, 5, 0, 0, 0, 0, 1000, 32), (64, 6, 0, 0, 0, 0, 1000, 32)]


def compile_emulation(folder, lanes):
    so = str(folder / ("bits_emulation_%d.so" % lanes))
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wno-attributes",
                           "-DXDROP_BITS_SHARED_MAX=%d" % lanes, "-o", so, os.path.join(HERE, "bits_emulation.cpp")])
    lib = ctypes.CDLL(so)
    lib.bits_emulate.restype = ctypes.c_longlong
    return lib


@pytest.fixture(scope="module")
def emulations(tmp_path_factory):
    """The form as it is, and with at most 2 lanes to an extension (above that it needs a whole warp)."""
    folder = tmp_path_factory.mktemp("bits")
    return {lanes: compile_emulation(folder, lanes) for lanes in (32, 2)}


def mutate(rng, s, err):
    out = []
    for ch in s:
        r = rng.random()
        if r < err * 0.2:
            out.append(rng.choice([c for c in "ACGT" if c != ch]))
        elif r < err * 0.7:
            out.append(ch + rng.choice("ACGT"))
        elif r >= err:
            out.append(ch)
    return "".join(out)


def sequences(rng, count, longest):
    """Pairs that overlap at several error rates, unrelated pairs, low-complexity
    pairs, and the smallest (empty, one base, equal, all mismatches)."""
    rand = lambda n: "".join(rng.choice("ACGT") for _ in range(n))
    out = [("", ""), ("A", ""), ("", "C"), ("A", "A"), ("A", "C"), ("AC" * 40, "AC" * 37), ("A" * 150, "C" * 150),
           ("A" * 90, "A" * 200), (rand(31), rand(33))]
    out += [(rand(longest), rand(longest)) for _ in range(14)]
    while len(out) < count:
        a = rand(rng.randint(1, longest))
        kind = rng.random()
        if kind < 0.5:
            b = mutate(rng, a, rng.choice([0.0, 0.05, 0.15, 0.3, 0.35]))
            if rng.random() < 0.3:
                b = b[:rng.randint(0, len(b))]
        elif kind < 0.8:
            b = rand(rng.randint(1, longest))
        else:
            unit = rand(rng.randint(1, 5))
            a, b = unit * (len(a) // len(unit)), mutate(rng, unit * (len(a) // len(unit) + 3), 0.1)
        out.append((a, b))
    return out


@pytest.mark.parametrize("case", range(len(CASES)))
def test_form_equals_oracle(emulations, case):
    form, nb, reserve, young, max_groups, pool, slots, lanes = CASES[case]
    emu = emulations[lanes]
    max_x = (1 << nb) - 5
    rng = random.Random(case)
    pairs = sequences(rng, 36, 300)
    reads = [s for p in pairs for s in p]
    ascii = np.frombuffer("".join(reads).encode(), dtype=np.uint8)
    offs = np.cumsum([0] + [len(r) for r in reads]).astype(np.int64)
    words, woffs, lens = dib.dibella_pack_reads(ascii, offs)
    n = len(pairs)
    copy = (((lens.astype(np.int64) + 15) // 16) + 3) // 4 * 4
    a0 = np.ascontiguousarray(woffs[0::2] * 16)
    b0 = np.ascontiguousarray((woffs[1::2] + copy[1::2]) * 16 + lens[1::2] - 1)
    la, lb = np.ascontiguousarray(lens[0::2]), np.ascontiguousarray(lens[1::2])
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    suspended = whole_warp = 0
    for X in sorted({1, 7, max_x // 2, max_x}):
        out = np.zeros((n, 4), dtype=np.int64)
        stats = np.zeros(4, dtype=np.int64)
        rc = emu.bits_emulate(form, p(words), ctypes.c_longlong(len(words)), p(a0), p(b0), p(la), p(lb), n, X,
                              reserve, young, max_groups, pool, slots, p(out), p(stats))
        assert rc == 0, "reads outside the store, or lanes out of step: %d" % rc
        suspended += int(stats[0])
        whole_warp += int(stats[3])
        assert stats[2] == 0  # no band here outgrows the whole-warp form
        for i, (a, b) in enumerate(pairs):
            assert tuple(out[i]) == oracle.extend(a, b, 1, -1, -1, X)[:4], (X, i, a, b)
    if reserve == 2 and nb == 5:  # unrelated sequences outgrow two lanes: these packings have to suspend
        assert suspended >= 3
    if lanes == 2:  # wide bands went to the whole-warp form, and some came back
        assert whole_warp > 5 and (not pool or suspended > 0)

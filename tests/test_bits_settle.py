"""Evaluated cells of the bit-sliced form between two layouts, per group (CPU).

A layout lasts as long as the band keeps its place: reads of 16 Mb that repeat
(TCCGGATGTT)n against the same with A and C, G and T exchanged keep a band of 280
to 285 cells in the middle of its window at X = 59 (the match table is symmetric),
9.5 G cells in 2^25 antidiagonals: more than 32 bits in the group, not in a lane."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("settle") / "bits_settle.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wno-attributes", "-o", so,
                           os.path.join(HERE, "bits_settle.cpp")])
    return ctypes.CDLL(so)


@pytest.mark.parametrize("length", [1, 2, 8, 16, 32])
@pytest.mark.parametrize("top", [1 << 20, 32 << 25])
def test_group_sums(lib, length, top):
    counts = np.random.default_rng(length).integers(top // 2, top, 32, dtype=np.uint32)
    sums = np.zeros(32, dtype=np.int64)
    lib.settle_sums(counts.ctypes.data_as(ctypes.c_void_p), length, sums.ctypes.data_as(ctypes.c_void_p))
    exp = counts.astype(np.int64).reshape(-1, length).sum(1) + 7
    assert np.array_equal(sums, np.repeat(exp, length))

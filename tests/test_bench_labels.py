"""bench.py names a batch's first launch by the form that ran, not by whether a schedule was passed (CPU)."""

import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("built_in,bits", [(True, {1, 7, 25, 59}), (False, set())])
def test_first_form_names(built_in, bits):
    names = bench.first_form_names(built_in, (0, 1, 7, 25, 59, 60))
    assert {X for X, name in names.items() if name == bench.BITS_FORM} == bits
    assert all(name == "narrow form" for X, name in names.items() if X not in bits)

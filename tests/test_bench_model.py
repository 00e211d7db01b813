"""CPU: bench.py's byte model of a level is what its kernels must move per point:
the key column for the split, and the scatter's columns and permutation in and
out. (Explicit subset ids are neither read nor moved by a level.)"""
from __future__ import annotations

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("d,want", [(1, 20), (3, 36), (8, 76), (16, 140)])
def test_bytes_of_a_level(d, want):
    assert bench.model_bytes_per_point_level(d) == want
    for sid_bytes, mode in ((0, 0), (1, 2), (2, 2)):
        assert want == (bench.bytes_per_point("k_part_count", d, sid_bytes, mode) +
                        bench.bytes_per_point("k_part_scatter", d, sid_bytes, mode))

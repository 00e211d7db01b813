"""The runs of tiles that the Fourier estimator sums (csrc/kdt_runs.h, compiled
for the host): a cell's runs are the same wherever the cell stands in the
step's tile list and however many CTAs walk that list, so that the order of a
cell's sums, and with it the tree, does not depend on scheduling."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_08288_gb300", "csrc")
WRAP = """#include "kdt_runs.h"
extern "C" uint32_t tiles(uint32_t n) { return kdt::run_tiles(n); }
extern "C" uint32_t start(uint32_t t, uint32_t i, uint32_t n, uint32_t len) { return kdt::run_start(t, i, n, len); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = tmp_path_factory.mktemp("runs")
    (out / "wrap.cpp").write_text(WRAP)
    subprocess.check_call(["g++", "-shared", "-fPIC", "-I", CSRC, "-o", str(out / "runs.so"), str(out / "wrap.cpp")])
    return ctypes.CDLL(str(out / "runs.so"))


def _runs(lib, cells, order, ctas, length):
    """Per cell, the (first tile, tiles) of every run that k_fourier_moments' CTAs sum, cells[k] tiles each."""
    tiles = [(c, i) for c in order for i in range(cells[c])]

    def start_from(t):
        return lib.start(t, tiles[t][1], cells[tiles[t][0]], length) if t < len(tiles) else len(tiles)

    runs = {c: [] for c in range(len(cells))}
    for k in range(ctas):
        begin, end = (start_from(j * len(tiles) // ctas) for j in (k, k + 1))
        first = begin
        for t in range(begin, end):
            c, i = tiles[t]
            if t + 1 == end or tiles[t + 1][0] != c or (i + 1) % length == 0:
                runs[c].append((tiles[first][1], t + 1 - first))
                first = t + 1
    return {c: sorted(r) for c, r in runs.items()}


@pytest.mark.parametrize("tree_tiles", [1, 40, 4096, 4097, 9000, 65536])
def test_a_cells_runs_do_not_depend_on_its_place(lib, tree_tiles):
    length = lib.tiles(tree_tiles)
    rng = np.random.default_rng(tree_tiles)
    total = min(tree_tiles, 6000)
    cuts = np.sort(rng.integers(0, total + 1, min(total, 50)))
    cells = [int(v) for v in np.diff(np.concatenate([[0], cuts, [total]])) if v > 0]
    want = {c: [(i, min(length, n - i)) for i in range(0, n, length)] for c, n in enumerate(cells)}
    for ctas in (1, 7, 304, 5000):
        for order in (np.arange(len(cells)), rng.permutation(len(cells)), rng.permutation(len(cells))):
            assert _runs(lib, cells, order.tolist(), ctas, length) == want


def test_a_root_has_a_bounded_number_of_runs(lib):
    for tiles in (1, 4095, 4096, 4097, 8193, 1 << 21):
        assert -(-tiles // lib.tiles(tiles)) <= 4096

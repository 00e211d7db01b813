"""GPU: the level step's small and large forms around where they change: few
and many segments (a CTA for every segment, or the lists by size), averages on
both sides of 8192 keys, cells of few and of very many tiles (one CTA per cell
for combine, count, scan and classify; a CTA or a warp for the scan), empty
and one-point segments, unbalanced cells, and the same trees together in one
batch, whose steps read their counts on the device. Bit for bit against the
oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_util import require_gpu
from paper_2201_08288_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _points(n, d, kind, seed):
    if kind == "uniform":
        return workloads.uniform(n, d, seed=seed)
    if kind == "ties":  # a coarse grid: cells that split unevenly or not at all
        return (np.random.default_rng(seed).integers(0, 5, (d, n)).astype(np.float32) ** 3) / 8
    return workloads.student_t_snapped(n, d, 3.0, 0.1, 256, seed=seed)


CASES = [
    (1_050_000, 3, "uniform", dict(r=8, depth=11)),              # 513 tiles in the root, 131,250 keys a segment
    (130_001, 2, "student", dict(r=1, leaf_size=64, max_levels=20)),
    (65_536, 3, "uniform", dict(r=8, depth=10)),                 # 8192 keys a segment
    (65_545, 3, "uniform", dict(r=8, depth=10)),                 # just above
    (40_000, 3, "student", dict(r=1216, leaf_size=32, max_levels=20)),
    (40_000, 3, "student", dict(r=1300, leaf_size=32, max_levels=20)),
    (9_000, 16, "uniform", dict(r=4096, leaf_size=64, max_levels=20)),
    (60_000, 3, "ties", dict(r=7, leaf_size=20, max_levels=24)),
    (60_000, 2, "ties", dict(r=3, depth=9, key_rule=1)),
    (250_007, 5, "student", dict(r=40, leaf_size=30, max_levels=20, key_rule=1)),
    (250_007, 8, "student", dict(r=64, depth=9, key_rule=1, combine_rule=1)),
    (300_001, 16, "uniform", dict(r=32, leaf_size=64, max_levels=20)),
]


def _same(g, o, what):
    assert g.levels == o.levels, what
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm), what
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32)), what
    assert np.array_equal(g.split_dims.cpu().numpy(), o.split_dims), what
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets), what


@pytest.mark.parametrize("case", range(len(CASES)))
def test_step_forms(case):
    from paper_2201_08288_gb300 import kdt
    n, d, kind, kw = CASES[case]
    x = _points(n, d, kind, case)
    _same(kdt.kdt_build(torch.from_numpy(x).cuda(), **kw), oracle.build_tree(x, **kw), str(CASES[case]))


def test_step_forms_in_one_batch():
    from paper_2201_08288_gb300 import kdt
    xs = [_points(n, d, kind, i) for i, (n, d, kind, _) in enumerate(CASES)]
    items = [dict(points=torch.from_numpy(x).cuda(), **c[3]) for x, c in zip(xs, CASES)]
    trees, status = kdt.kdt_build_batched(items)
    assert status == [0] * len(CASES)
    for t, x, c in zip(trees, xs, CASES):
        _same(t, oracle.build_tree(x, **c[3]), str(c))


WIDE = [
    (300_007, 3, "uniform", dict(r=1, leaf_size=40, max_levels=20)),
    (800_007, 2, "student", dict(r=3, depth=8)),
    (1_048_576, 3, "student", dict(r=4, depth=7)),          # 262,144 keys a segment
    (1_048_575, 3, "student", dict(r=4, depth=7)),          # just below
    (600_001, 1, "ties", dict(r=2, depth=5)),
    (900_001, 5, "student", dict(r=3, depth=6, key_rule=1)),
    (2_900, 2, "uniform", dict(r=2, depth=3)),              # beside large trees: no room for a histogram per segment
]


@pytest.mark.parametrize("case", range(len(WIDE)))
def test_several_ctas_per_segment(case):
    from paper_2201_08288_gb300 import kdt
    n, d, kind, kw = WIDE[case]
    x = _points(n, d, kind, 50 + case)
    _same(kdt.kdt_build(torch.from_numpy(x).cuda(), **kw), oracle.build_tree(x, **kw), str(WIDE[case]))


def test_several_ctas_per_segment_in_one_batch():
    from paper_2201_08288_gb300 import kdt
    xs = [_points(n, d, kind, 50 + i) for i, (n, d, kind, _) in enumerate(WIDE)]
    trees, status = kdt.kdt_build_batched([dict(points=torch.from_numpy(x).cuda(), **c[3]) for x, c in zip(xs, WIDE)])
    assert status == [0] * len(WIDE)
    for t, x, c in zip(trees, xs, WIDE):
        _same(t, oracle.build_tree(x, **c[3]), str(c))


def test_several_ctas_for_unequal_subsets():
    """Explicit ids, one subset nearly empty: its segment takes the path by size."""
    from paper_2201_08288_gb300 import kdt
    n = 1_100_007
    x = _points(n, 3, "student", 90)
    sid = (np.random.default_rng(1).random(n) < 0.5).astype(np.uint8)
    sid[::3001] = 2
    kw = dict(r=4, subset_mode=2, depth=8)  # subset 3 is empty
    g = kdt.kdt_build(torch.from_numpy(x).cuda(), sid=torch.from_numpy(sid).cuda(), **kw)
    _same(g, oracle.build_tree(x, sid=sid, **kw), "unequal")

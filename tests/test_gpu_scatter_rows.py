"""GPU: the children's subset offsets that the scatter derives from the cell's
own, and the subsets that the subtree kernel takes from them: few and many
subsets, empty ones and one that holds nearly everything, fewer and more
subsets than a small cell has points (rows kept, ids gathered), 8- and 16-bit
ids, every compiled coordinate count and one without, contiguous subsets of
sizes that do not divide n. Bit for bit against the oracle."""
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


def _check(pts, gpu_sid, sid, **kw):
    from paper_2201_08288_gb300 import kdt
    g = kdt.kdt_build(torch.from_numpy(pts).cuda(), sid=gpu_sid, **kw)
    o = oracle.build_tree(pts, sid=sid, **kw)
    assert g.levels == o.levels
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32))
    assert np.array_equal(g.split_dims.cpu().numpy(), o.split_dims)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)


@pytest.mark.parametrize("n,d,r,skew,rule", [
    (20_011, 3, 1, 0.0, 1), (20_011, 3, 2, 0.0, 0), (50_003, 8, 255, 0.0, 1), (50_003, 2, 256, 0.9, 0),
    (50_003, 16, 257, 0.0, 1), (50_003, 5, 700, 0.5, 0), (30_011, 3, 1300, 0.0, 0), (30_011, 8, 4096, 0.99, 1),
    (4097, 16, 300, 0.0, 0), (2049, 64, 33, 0.0, 1)])
def test_explicit_ids(n, d, r, skew, rule):
    rng = np.random.default_rng(n + r)
    pts = workloads.student_t_snapped(n, d, 3.0, 0.1, 256, seed=r)
    sid = rng.integers(0, r, n)
    sid[rng.random(n) < skew] = r // 2
    sid[sid == r // 3] = r - 1  # an empty subset
    sid = sid.astype(np.uint8 if r <= 256 else np.uint16)
    gpu_sid = torch.from_numpy(sid if r <= 256 else sid.view(np.int16)).cuda()
    _check(pts, gpu_sid, sid, r=r, subset_mode=2, leaf_size=20, max_levels=20, key_rule=rule)


@pytest.mark.parametrize("n,r", [(100_003, 1), (100_003, 3), (100_003, 64), (99_991, 4096), (70_001, 1023), (4095, 4096)])
@pytest.mark.parametrize("mode", [0, 1])
def test_ids_from_the_index(n, r, mode):
    pts = workloads.gaussian_mixture(n, 3, 16, 0.05, seed=r)
    _check(pts, None, None, r=r, subset_mode=mode, leaf_size=24, max_levels=22)


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("d", [1, 4, 6, 7, 9, 12, 13])
def test_coordinate_counts(d, rule):
    n = 30_000 + 77 * d
    pts = workloads.student_t_snapped(n, d, 3.0, 0.1, 256, seed=d)
    sid = np.random.default_rng(d).integers(0, 40, n).astype(np.uint8)
    _check(pts, torch.from_numpy(sid).cuda(), sid, r=40, subset_mode=2, leaf_size=16, max_levels=20, key_rule=rule)

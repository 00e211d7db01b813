"""GPU: leaves of 257 to 4096 points, sorted by a CTA in buckets or, where the
indices are so uneven that a bucket overflows, by radix; few and many leaves,
one tree and several together. Bit for bit against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_util import require_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _cloud(n, depth, order):
    rng = np.random.default_rng(n + depth)
    x = rng.random((2, n)).astype(np.float32)
    if order == "sorted":
        x[0] = x[1] = np.sort(x[0])
    elif order == "burst":  # the first leaf: half of it one stretch of indices, half spread over the whole range
        leaf = n >> depth
        x[0] += 1.0
        x[0, :leaf // 2] -= 1.0
        x[0, rng.choice(np.arange(leaf // 2, n), leaf - leaf // 2, replace=False)] -= 1.0
        x[1] = x[0]
    return x


CASES = [(2 * 257, 1, "any"), (4 * 4095, 2, "any"), (2 * 4096, 1, "sorted"), (300 * 1024, 10, "any"),
         (1_000_003, 9, "any"), (900_000, 8, "burst"), (700, 1, "burst"), (3 * 512 + 1, 2, "any")]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_middle_leaves(case):
    from paper_2201_08288_gb300 import kdt
    n, depth, order = CASES[case]
    x = _cloud(n, depth, order)
    kw = dict(r=16, subset_mode=0, depth=depth)
    g, o = kdt.kdt_build(torch.from_numpy(x).cuda(), **kw), oracle.build_tree(x, **kw)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)


def test_middle_leaves_of_several_trees():
    from paper_2201_08288_gb300 import kdt
    xs = [_cloud(*c) for c in CASES]
    items = [dict(points=torch.from_numpy(x).cuda(), r=16, depth=c[1]) for x, c in zip(xs, CASES)]
    trees, status = kdt.kdt_build_batched(items)
    assert status == [0] * len(CASES)
    for t, x, c in zip(trees, xs, CASES):
        o = oracle.build_tree(x, r=16, subset_mode=0, depth=c[1])
        assert np.array_equal(t.perm.cpu().numpy().view(np.uint32), o.perm), c

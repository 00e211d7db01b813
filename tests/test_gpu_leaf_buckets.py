"""GPU: the order of leaves too large for one CTA's radix sort: sizes around
the bounds of the bucket pass (4096, 54,272 points), indices that fill a
narrow range, and indices so unevenly spread that a bucket overflows and the
leaf goes through the global passes. The permutation inside a leaf is
ascending; bit for bit against the oracle."""
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


def _burst(n, leaf, rng):
    """One coordinate whose smallest values (about a leaf of them) are those of one stretch of indices and of some
    spread over the whole range."""
    x = rng.random(n) + 1.0
    x[:leaf // 2] -= 1.0
    x[rng.choice(np.arange(leaf // 2, n), leaf - leaf // 2, replace=False)] -= 1.0
    return x


@pytest.mark.parametrize("n,depth,order", [
    (2 * 4096, 1, "any"), (2 * 4097, 1, "any"), (8 * 5000 + 3, 3, "any"), (2 * 54_272, 1, "any"),
    (2 * 54_272 + 2, 1, "any"), (200_003, 2, "sorted"), (800_001, 4, "burst"), (300_001, 1, "any")])
def test_large_leaves(n, depth, order):
    from paper_2201_08288_gb300 import kdt
    rng = np.random.default_rng(n)
    x = rng.random((2, n)).astype(np.float32)
    if order == "sorted":  # every leaf holds a contiguous range of indices
        x[0] = np.sort(x[0])
        x[1] = x[0]
    elif order == "burst":
        x[0] = x[1] = _burst(n, n >> depth, rng)
    kw = dict(r=64, subset_mode=0, depth=depth)
    g = kdt.kdt_build(torch.from_numpy(x).cuda(), **kw)
    o = oracle.build_tree(x, **kw)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)

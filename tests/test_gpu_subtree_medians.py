"""GPU: the subtree kernel's segment medians by segment size: rank counting (up
to 32 points), a warp's network (to 64), bit by bit in registers (to 512) and
by radix histogram above, around every bound, with distinct keys, ties, signed
zeros and infinities; narrow and wide shapes, both key rules. Bit for bit
against the oracle."""
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


def _points(n, d, kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "distinct":
        return rng.standard_normal((d, n)).astype(np.float32)
    x = (rng.integers(-3, 4, (d, n)) / 4).astype(np.float32)  # ties
    x[x == 0] = np.where(rng.random((x == 0).sum()) < 0.5, -0.0, 0.0)
    x[rng.random((d, n)) < 0.01] = np.inf
    x[rng.random((d, n)) < 0.01] = -np.inf
    return x


@pytest.mark.parametrize("w", [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1024])
@pytest.mark.parametrize("kind", ["distinct", "ties"])
@pytest.mark.parametrize("d,rule", [(2, 0), (5, 1), (12, 0)])
def test_segment_sizes(w, kind, d, rule):
    from paper_2201_08288_gb300 import kdt
    r = max(1, min(7, 1270 // w))  # at most 1270 points: one cell of either shape
    n = r * w
    x = _points(n, d, kind, w)
    kw = dict(r=r, subset_mode=0, leaf_size=3, max_levels=24, key_rule=rule)
    g, o = kdt.kdt_build(torch.from_numpy(x).cuda(), **kw), oracle.build_tree(x, **kw)
    assert g.levels == o.levels
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32))
    assert np.array_equal(g.split_dims.cpu().numpy(), o.split_dims)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)

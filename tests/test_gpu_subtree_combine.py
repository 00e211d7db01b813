"""GPU: the subtree kernel's weighted median of the segment medians on both sides
of its line (up to 16 subsets by a thread per segment, more by a warp per cell):
segments of very different sizes, equal medians, empty subsets, both combine
rules, all three shapes. Bit for bit against the oracle."""
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


@pytest.mark.parametrize("r", [1, 2, 3, 15, 16, 17, 33])
@pytest.mark.parametrize("n,d", [(40, 2), (1000, 3), (1900, 12), (9000, 4)])
@pytest.mark.parametrize("combine", [0, 1])
@pytest.mark.parametrize("ties", [False, True])
def test_combine(r, n, d, combine, ties):
    from paper_2201_08288_gb300 import kdt
    rng = np.random.default_rng(r + n)
    x = (rng.integers(-4, 5, (d, n)) / 2 if ties else rng.standard_normal((d, n))).astype(np.float32)
    sid = (rng.random(n) ** 4 * r).astype(np.uint8)
    sid[sid == r // 2] = 0  # an empty subset where there are several
    kw = dict(r=r, subset_mode=2, depth=9, combine_rule=combine)
    g = kdt.kdt_build(torch.from_numpy(x).cuda(), sid=torch.from_numpy(sid).cuda(), **kw)
    o = oracle.build_tree(x, sid=sid, **kw)
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32))
    assert np.array_equal(g.split_dims.cpu().numpy(), o.split_dims)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)

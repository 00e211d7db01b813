"""GPU: many searches at once, which go a thread per query where they are short,
against the same searches a few thousand at a time, which go a warp each: the
same answers, bit for bit. Leaves of one to many points, empty ones, one point in
all; short and long searches mixed in a warp; equal distances; infinities and NaN
on both sides; lists shorter than what they list; ragged numbers of queries on
both sides of the line."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import require_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
FEW = 4096  # queries of a call that always go a warp each


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _tree(n, d, kind, leaf, seed=1):
    from paper_2201_08288_gb300 import kdt
    rng = np.random.default_rng(seed + n + d)
    x = rng.standard_normal((d, n)).astype(np.float32)
    if kind == "ties":
        x = np.round(x * 2) / 2
    if kind == "inf" and n > 20:
        x[0, ::9], x[d - 1, 1::13] = np.inf, -np.inf
    X = torch.from_numpy(x).cuda()
    kw = dict(depth=-leaf) if leaf < 0 else dict(leaf_size=leaf, max_levels=22)
    return x, X, kdt.kdt_build(X, r=4, key_rule=1, **kw)


def _queries(x, nq, kind, seed=2):
    rng = np.random.default_rng(seed)
    n = x.shape[1]
    q = x[:, rng.integers(0, n, nq)]
    near = rng.random(nq) < 0.5
    q = np.where(near, q + (0.3 * rng.standard_normal(q.shape)).astype(np.float32), q).astype(np.float32)
    if kind == "inf":
        q[0, rng.random(nq) < 0.01] = np.inf
        q[-1, rng.random(nq) < 0.01] = np.nan
    return np.ascontiguousarray(q)


CASES = [(1, 1, "normal", 1), (40, 2, "normal", 1), (3000, 3, "normal", 1), (3000, 3, "normal", 4), (3000, 3, "ties", 2),
         (3000, 2, "inf", 1), (3000, 3, "normal", 60), (700, 17, "normal", 2), (2000, 3, "normal", -14),
         (5000, 1, "normal", 2), (400, 3, "inf", 8)]


@pytest.mark.parametrize("n,d,kind,leaf", CASES)
@pytest.mark.parametrize("nq", [32_767, 32_768, 70_001, 1_200_001])
def test_nearest(n, d, kind, leaf, nq):
    from paper_2201_08288_gb300 import kdt
    x, X, t = _tree(n, d, kind, leaf)
    Q = torch.from_numpy(_queries(x, nq, kind)).cuda()
    idx, d2 = kdt.kdt_query_knn(X, t, Q, 1)
    some = [0, nq - FEW] if nq > 100_000 else range(0, nq, FEW)
    for a in some:
        wi, wd = kdt.kdt_query_knn(X, t, Q[:, a:a + FEW].contiguous(), 1)
        assert torch.equal(idx[a:a + FEW], wi)
        assert torch.equal(d2[a:a + FEW].view(torch.int64), wd.view(torch.int64))


@pytest.mark.parametrize("n,d,kind,leaf", CASES)
@pytest.mark.parametrize("nq,cap", [(32_767, 3), (32_768, 40), (70_001, 0), (1_200_001, 2)])
def test_boxes(n, d, kind, leaf, nq, cap):
    from paper_2201_08288_gb300 import kdt
    x, X, t = _tree(n, d, kind, leaf)
    q = _queries(x, nq, kind)
    rng = np.random.default_rng(3)
    half = (0.02 + 0.1 * rng.random(nq)).astype(np.float32)
    half[rng.random(nq) < 0.002] = 50.0  # everything, among short ones
    half[rng.random(nq) < 0.02] = -1.0   # nothing
    if nq > 65_536:
        half[:20_000] = 1.5              # stretches of long searches
    L, H = torch.from_numpy(q - half).cuda(), torch.from_numpy(q + half).cuda()
    counts, lists = kdt.kdt_query_box(X, t, L, H, list_cap=cap)
    some = [0, 18_000, nq - FEW] if nq > 100_000 else range(0, nq, FEW)
    for a in some:
        wc, wl = kdt.kdt_query_box(X, t, L[:, a:a + FEW].contiguous(), H[:, a:a + FEW].contiguous(), list_cap=cap)
        assert torch.equal(counts[a:a + FEW], wc)
        if cap:
            assert torch.equal(lists[a:a + FEW], wl)

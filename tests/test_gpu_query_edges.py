"""GPU: the warp-per-query searches at the sizes and values where they can go
wrong: leaves of 1, 31..33 and more points than a round of 32 lanes takes, one
to 64 coordinates, k at both ends, magnitudes whose float squares underflow or
overflow (a point is measured in float before it is measured in double),
infinities, and queries whose distances are no numbers. All comparisons are
exact: the double distances are a fixed function of the inputs."""
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


def _cloud(n, d, scale, seed):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((d, n)) * scale).astype(np.float32)
    x[:, rng.integers(0, n, n // 8)] = x[:, rng.integers(0, n, n // 8)]  # duplicates: ties in the distance
    return x


def _nearest(x, q, k):
    with np.errstate(over="ignore"):
        return oracle.nearest(x, q, k)


@pytest.mark.parametrize("n,d,leaf,scale", [
    (1, 1, 1, 1.0), (31, 2, 1, 1.0), (700, 3, 31, 1.0), (700, 3, 32, 1e-21), (700, 3, 33, 3e18), (2000, 9, 100, 1.0),
    (1500, 64, 40, 1.0), (1500, 17, 8, 1e-30), (900, 8, 500, 1e37), (40, 3, 5, 1e-25), (64, 2, 64, 2e18)])
@pytest.mark.parametrize("k", [1, 7, 8, 32])
def test_knn_at_edges(n, d, leaf, scale, k):
    from paper_2201_08288_gb300 import kdt
    x = _cloud(n, d, scale, n + d)
    if n > 500:  # points at infinity: at an infinite distance from every finite query
        x[0, 3], x[d - 1, 5] = np.inf, -np.inf
    X = torch.from_numpy(x).cuda()
    t = kdt.kdt_build(X, r=4, leaf_size=leaf, max_levels=20)
    rng = np.random.default_rng(7)
    q = np.concatenate([_cloud(max(n, 9), d, scale, 5)[:, :9], x[:, rng.integers(6, n, 9) if n > 6 else [0] * 9]], axis=1)
    idx, d2 = kdt.kdt_query_knn(X, t, torch.from_numpy(q).cuda(), k)
    idx, d2 = idx.cpu().numpy().view(np.uint32), d2.cpu().numpy()
    m = min(k, n)
    for j in range(q.shape[1]):
        wi, wd = _nearest(x, q[:, j], m)
        assert np.array_equal(d2[j, :m], wd), f"query {j} distances"
        assert np.array_equal(idx[j, :m], wi.astype(np.uint32)), f"query {j}"
        assert np.all(idx[j, m:] == 0xFFFFFFFF) and np.all(np.isinf(d2[j, m:]))


def _serial_knn(x, tree, q, k):
    """The list that insertion in visiting order gives when distances are in no order (NaN). A NaN coordinate of the
    query has no side; the search takes it to the left, as it always has."""
    perm, vals, dims, offs = (a.cpu().numpy() for a in (tree.perm, tree.split_vals, tree.split_dims, tree.node_offsets))
    x, q = x.astype(np.float64), q.astype(np.float64)
    best, nbest = [(np.inf, 0xFFFFFFFF)] * k, 0
    stack = [(0, 0.0)]
    while stack:
        h, bound = stack.pop()
        if nbest == k and bound > best[-1][0]:
            continue
        lv = int(np.log2(h + 1))
        if lv < tree.levels and dims[h] >= 0:
            t = dims[h]
            qk, mk = oracle.order_keys(np.array([q[t], vals[h]], np.float32))
            near, far = (2 * h + 1, 2 * h + 2) if qk <= mk or np.isnan(q[t]) else (2 * h + 2, 2 * h + 1)
            stack += [(far, np.fmax(bound, (q[t] - np.float64(vals[h])) ** 2)), (near, bound)]
            continue
        leaf = (h - (2 ** lv - 1)) << (tree.levels - lv)
        for i in perm[offs[leaf]:offs[leaf + 1]]:
            d2 = 0.0
            for j in range(len(q)):
                d2 += (x[j, i] - q[j]) ** 2
            e = (d2, int(i))
            if nbest == k and not e < best[-1]:
                continue
            pos, nbest = (nbest, nbest + 1) if nbest < k else (k - 1, k)
            for j in range(k - 1, 0, -1):
                if j <= pos and e < best[j - 1]:
                    best[j] = best[j - 1]
                    pos = j - 1
            best[pos] = e
    return best


@pytest.mark.filterwarnings("ignore::RuntimeWarning")
@pytest.mark.parametrize("k", [1, 6, 32])
def test_knn_with_distances_that_are_no_numbers(k):
    from paper_2201_08288_gb300 import kdt
    x = _cloud(600, 3, 1.0, 3)
    x[0, ::7] = np.inf
    x[1, ::11] = -np.inf
    X = torch.from_numpy(x).cuda()
    t = kdt.kdt_build(X, r=4, leaf_size=20, max_levels=20)
    q = _cloud(12, 3, 1.0, 4)
    q[0, :4], q[1, 4:6], q[2, 6:9] = np.inf, -np.inf, np.nan
    idx, d2 = kdt.kdt_query_knn(X, t, torch.from_numpy(q).cuda(), k)
    idx, d2 = idx.cpu().numpy().view(np.uint32), d2.cpu().numpy()
    for j in range(q.shape[1]):
        want = _serial_knn(x, t, q[:, j], k)
        assert idx[j].tolist() == [i for _, i in want], f"query {j}"
        assert np.array_equal(d2[j], [v for v, _ in want], equal_nan=True), f"query {j}"


@pytest.mark.parametrize("n,d,leaf", [(1, 1, 1), (40, 2, 33), (900, 3, 31), (900, 5, 64), (900, 64, 100)])
@pytest.mark.parametrize("cap", [1, 33, 1000])
def test_box_lists_keep_the_order_of_the_leaves(n, d, leaf, cap):
    from paper_2201_08288_gb300 import kdt
    x = _cloud(n, d, 1.0, 11)
    X = torch.from_numpy(x).cuda()
    t = kdt.kdt_build(X, r=2, leaf_size=leaf, max_levels=20)
    rng = np.random.default_rng(5)
    a, b = x[:, rng.integers(0, n, 20)], x[:, rng.integers(0, n, 20)]
    lo, hi = np.minimum(a, b) - np.float32(0.5), np.maximum(a, b) + np.float32(0.5)
    lo[:, 0], hi[:, 0] = -np.inf, np.inf
    lo[0, 1], hi[0, 1] = 1.0, -1.0
    counts, lists = kdt.kdt_query_box(X, t, torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda(), list_cap=cap)
    counts, lists, perm = counts.cpu().numpy(), lists.cpu().numpy(), t.perm.cpu().numpy()
    for q in range(20):
        inside = set(oracle.box_members(x, lo[:, q], hi[:, q]).tolist())
        want = [i for i in perm if i in inside]
        assert counts[q] == len(want), f"box {q}"
        assert lists[q, :min(cap, len(want))].tolist() == want[:cap], f"box {q}"


@pytest.mark.parametrize("k", [1, 8, 31, 32])
def test_knn_with_many_equal_distances(k):
    """More points at one distance than the list of 32 holds: the smaller indices win."""
    from paper_2201_08288_gb300 import kdt
    rng = np.random.default_rng(2)
    x = rng.integers(-2, 3, (3, 4000)).astype(np.float32)
    X = torch.from_numpy(x).cuda()
    t = kdt.kdt_build(X, r=4, leaf_size=33, max_levels=24)
    q = np.concatenate([x[:, :10], x[:, :10] + np.float32(0.5)], axis=1)
    idx, d2 = kdt.kdt_query_knn(X, t, torch.from_numpy(q).cuda(), k)
    for j in range(q.shape[1]):
        wi, wd = _nearest(x, q[:, j], k)
        assert np.array_equal(d2[j].cpu().numpy(), wd) and np.array_equal(idx[j].cpu().numpy(), wi), f"query {j}"

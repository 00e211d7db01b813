"""GPU: level steps launched ahead of their counts (trees built alone): splits
far from the middle, so that cells are left when the steps sure to be needed are
done; ties that end the tree early, so that steps find no cells; caps on the
levels; few, large segments; the estimator's steps. Bit for bit against the
oracle (the estimator's splits against its evaluation on the host)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_util import gpu_build, require_gpu
from test_gpu_fourier import check_tree

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
KDT_ERR_LEVEL_CAP = 7


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _points(kind, n, d):
    rng = np.random.default_rng(n + d)
    x = rng.standard_normal((d, n)).astype(np.float32)
    if kind == "skewed":  # subsets (blocks of the index) of very different places: splits far from the middle
        x += (np.arange(n) / n > 0.45).astype(np.float32) * np.float32(50) * np.arange(n, dtype=np.float32) ** 2 / n
    elif kind == "few":  # 4 values a coordinate: leaf cells early
        x = rng.integers(0, 4, (d, n)).astype(np.float32)
    elif kind == "one":  # the widest coordinate alone decides, the rest is constant
        x[1:] = 1.0
    return x


@pytest.mark.parametrize("kind", ["normal", "skewed", "few", "one"])
@pytest.mark.parametrize("n,d,r,mode,rule,kw", [
    (20_000, 3, 5, 1, 0, dict(leaf_size=30, max_levels=25)), (150_001, 2, 11, 1, 1, dict(leaf_size=200, max_levels=25)),
    (150_001, 2, 64, 0, 1, dict(leaf_size=7, max_levels=5)), (300_000, 1, 3, 1, 0, dict(leaf_size=9000, max_levels=20)),
    (600_011, 4, 2, 1, 0, dict(depth=9)), (100_003, 12, 900, 1, 1, dict(depth=4)), (40_000, 3, 1, 1, 1, dict(depth=1))])
def test_steps_ahead(kind, n, d, r, mode, rule, kw):
    from paper_2201_08288_gb300 import kdt
    x = _points(kind, n, d)
    kw = dict(kw, r=r, subset_mode=mode, key_rule=rule)
    X = torch.from_numpy(x).cuda()
    try:
        o = oracle.build_tree(x, **kw)
    except oracle.OracleError:  # more levels than the cap: refused for that, and a build with room works after it
        with pytest.raises(kdt.KdtError) as err:
            kdt.kdt_build(X, **kw)
        assert err.value.status == KDT_ERR_LEVEL_CAP
        kw.update(max_levels=25, leaf_size=max(kw["leaf_size"], 200))
        o = oracle.build_tree(x, **kw)
    g = kdt.kdt_build(X, **kw)
    assert g.levels == o.levels
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32))
    assert np.array_equal(g.split_dims.cpu().numpy(), o.split_dims)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)


@pytest.mark.parametrize("depth", [1, 8, 13])
def test_estimator(depth):
    x = np.clip(np.random.default_rng(5).random((3, 50_000), dtype=np.float32) ** 3, 1e-6, 1 - 1e-6)
    check_tree(x, gpu_build(x, depth=depth, fourier_j=9), 9)


def test_a_traced_build_states_its_points():
    from paper_2201_08288_gb300 import kdt
    x = torch.rand(3, 70_001, device="cuda")
    kw = dict(r=8, subset_mode=0, depth=12)
    a = kdt.kdt_build(x, **kw)
    kdt.kdt_trace_enable(True)
    try:
        kdt.kdt_trace_read(True)
        b = kdt.kdt_build(x, **kw)
        units = {k: v[2] for k, v in kdt.kdt_trace_read(True).items()}
    finally:
        kdt.kdt_trace_enable(False)
    assert units["k_subtree"] == 70_001  # every point ends in a small cell
    assert torch.equal(a.perm, b.perm) and torch.equal(a.split_vals, b.split_vals)

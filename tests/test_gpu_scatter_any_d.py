"""GPU: the scatter for coordinate counts without a kernel of their own. Its
sub-tiles are parts of a tile that the buffers have room for, of another size
for every few d: trees around those sizes, bit for bit against the oracle; and
no d costs much more per column than one just below it (sub-tiles of half the
size had 2,000,003 points in 40 coordinates take 1.32 times as long)."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from gpu_util import assert_same_tree, gpu_build, require_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("d,n", [(9, 20_480), (10, 26_001), (13, 9_217), (17, 12_289), (23, 7_001), (29, 8_191),
                                 (35, 6_145), (47, 8_193), (64, 5_003)])
@pytest.mark.parametrize("rule,mode", [(0, 0), (1, 2), (1, 1)])
def test_any_d(d, n, rule, mode):
    rng = np.random.default_rng(d)
    x = rng.standard_normal((d, n)).astype(np.float32)
    x[:, rng.random(n) < 0.3] = np.float32(0.5)  # cells of unequal sizes
    sid = rng.integers(0, 37, n).astype(np.uint8) if mode == 2 else None
    kw = dict(r=37, subset_mode=mode, key_rule=rule, depth=8)
    assert_same_tree(gpu_build(x, sid=sid, **kw), oracle.build_tree(x, sid=sid, **kw), f"d {d}")


def test_together_in_one_batch():
    from paper_2201_08288_gb300 import kdt
    rng = np.random.default_rng(1)
    xs = [rng.standard_normal((d, 7000 + 13 * d)).astype(np.float32) for d in (9, 23, 35, 3, 64)]
    kw = dict(r=20, leaf_size=40, max_levels=20, key_rule=1)
    trees, status = kdt.kdt_build_batched([dict(points=torch.from_numpy(x).cuda(), **kw) for x in xs])
    assert status == [0] * len(xs)
    for t, x in zip(trees, xs):
        g = oracle.Tree(t.perm.cpu().numpy().view(np.uint32), t.split_vals.cpu().numpy(), t.split_dims.cpu().numpy(),
                        t.node_offsets.cpu().numpy(), t.levels)
        assert_same_tree(g, oracle.build_tree(x, **kw), f"d {len(x)}")


def test_time_per_column_has_no_jump():
    from paper_2201_08288_gb300 import kdt
    n = 1_000_003

    def per_column(d):
        x = torch.randn((d, n), device="cuda", generator=torch.Generator(device="cuda").manual_seed(d))
        best = float("inf")
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            kdt.kdt_build(x, r=64, leaf_size=64, max_levels=20, key_rule=1)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best / d

    assert per_column(36) < 1.35 * per_column(33)  # 1.7 and more with half the sub-tile

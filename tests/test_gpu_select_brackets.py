"""GPU: medians of listed segments by a warp's brackets, by segment size: around
each change of the sample, the rooms after a pass and the last sort; keys for
which the sample misleads (sorted, periodic), thins out badly (few values, one
value for most) or not at all (all equal), infinities and signed zeros. One
level of many contiguous subsets, bit for bit against the oracle."""
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


def _keys(kind, r, w, rng):
    n = r * w
    if kind == "sorted":
        return np.sort(rng.standard_normal((r, w)), axis=1)[:, :: 1 if w % 2 else -1].reshape(-1)
    if kind == "periodic":  # a sample at even distances sees a few values only
        return (np.arange(n) % 32) * 1.5 + rng.integers(0, 2, n)
    if kind == "few":
        return rng.integers(-2, 3, n) / 2
    if kind == "mostly":
        return np.where(rng.random(n) < 0.9, 0.5, rng.standard_normal(n))
    if kind == "equal":
        return np.full(n, -3.25)
    x = rng.standard_normal(n)
    if kind == "special":
        x[rng.random(n) < 0.2] = np.inf
        x[rng.random(n) < 0.2] = -np.inf
        z = rng.random(n) < 0.3
        x[z] = np.where(rng.random(z.sum()) < 0.5, 0.0, -0.0)
    return x


@pytest.mark.parametrize("w", [65, 127, 128, 129, 255, 256, 257, 511, 777, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096])
@pytest.mark.parametrize("kind", ["normal", "sorted", "periodic", "few", "mostly", "equal", "special"])
def test_sizes(w, kind):
    from paper_2201_08288_gb300 import kdt
    r = 1250  # more segments than get a CTA each
    x = _keys(kind, r, w, np.random.default_rng(w)).astype(np.float32)[None, :]
    kw = dict(r=r, subset_mode=1, depth=1)
    g, o = kdt.kdt_build(torch.from_numpy(x).cuda(), **kw), oracle.build_tree(x, **kw)
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32))
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)

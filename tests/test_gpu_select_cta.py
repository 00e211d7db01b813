"""GPU: the radix select of a CTA per segment by the number of segments (1024
threads while two CTAs per SM take them all, then 512, then 256 by the tuning)
and the digit width, around both lines, for segments with ties, infinities and
unaligned starts. Bit for bit against the oracle."""
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


@pytest.mark.parametrize("per_sm,more", [(0, 1), (0, 33), (2, 0), (2, 1), (8, 0), (8, 1)])
@pytest.mark.parametrize("bits", [8, 11])
def test_segments(per_sm, more, bits):
    from paper_2201_08288_gb300 import kdt
    r = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    w = 8193 if r > 8 else 30_001
    rng = np.random.default_rng(r)
    x = (rng.standard_normal(r * w) * np.repeat(rng.choice([1e-3, 1.0, 1e20], r), w)).astype(np.float32)
    x[rng.random(r * w) < 0.05] = np.inf
    x[rng.random(r * w) < 0.05] = -np.inf
    x[rng.random(r * w) < 0.2] = 0.5
    x = x[None, :]
    kw = dict(r=r, subset_mode=1, depth=1)
    kdt.set_tuning(dict(kdt.tuning_default(), digit_bits=bits))
    try:
        g = kdt.kdt_build(torch.from_numpy(x).cuda(), **kw)
    finally:
        kdt.set_tuning(None)
    o = oracle.build_tree(x, **kw)
    assert np.array_equal(g.split_vals.cpu().numpy().view(np.uint32), o.split_vals.view(np.uint32))
    assert np.array_equal(g.perm.cpu().numpy().view(np.uint32), o.perm)
    assert np.array_equal(g.node_offsets.cpu().numpy(), o.node_offsets)

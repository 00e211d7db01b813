"""Problems that kdt_build_noalloc's fixed 64 MiB have room for (host only: the
size of their workspace), near that limit: deep and shallow trees, both kinds of
depth, explicit ids, the estimator."""
from __future__ import annotations

import ctypes

import pytest


@pytest.mark.parametrize("n,d,kw", [
    (1_766_122, 2, dict(r=2, subset_mode=0, leaf_size=32, max_levels=16, key_rule=1)),
    (743_241, 5, dict(r=8, subset_mode=2, sid_ptr=4096, sid_bytes=1, leaf_size=32, max_levels=18, key_rule=1)),
    (1_525_760, 1, dict(r=256, subset_mode=1, leaf_size=1, max_levels=18, key_rule=1)),
    (515_129, 8, dict(r=1, subset_mode=1, leaf_size=1, max_levels=18, key_rule=1)),
    (51_840, 7, dict(r=32, subset_mode=2, sid_ptr=4096, sid_bytes=1, depth=16, fourier_j=8)),
    (2_573_998, 1, dict(r=64, subset_mode=0, depth=12))])
def test_fits_the_fixed_scratch(n, d, kw):
    from paper_2201_08288_gb300 import kdt
    lib = kdt.load_library()
    kw = dict(kw)
    j = kw.pop("fourier_j", 0)
    p = kdt.make_params(n, d, **kw)
    p.fourier_j = j
    need = ctypes.c_size_t(0)
    assert lib.kdt_workspace_size(ctypes.byref(p), ctypes.byref(need)) == 0
    assert need.value <= 64 << 20

"""GPU: the Fourier split's division of a cell's work: harmonic counts around the
sizes where its threads' parts meet (a candidate per half warp, the last two
warps free for the next midpoints up to J = 27, a thread per candidate and
harmonic), run records around whole chunks of 32, cells whose bounds are the
interval's ends and inner ones. Every node against the estimator on the host."""
from __future__ import annotations

import pytest

from gpu_util import gpu_build, require_gpu
from paper_2201_08288_gb300 import workloads
from test_gpu_fourier import check_tree

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("J", [1, 2, 7, 8, 15, 16, 23, 24, 27, 28, 31, 32])
def test_harmonics(J):
    n = 9000 + J
    pts = workloads.uniform_open(n, 2, seed=J)
    check_tree(pts, gpu_build(pts, depth=5, fourier_j=J), J)


@pytest.mark.parametrize("tiles,more", [(31, 0), (32, 0), (32, 1), (63, 5), (64, 0), (64, 1), (304, 0), (700, 3)])
def test_runs(tiles, more):
    n = tiles * 2048 + more
    pts = workloads.uniform_open(n, 1, seed=tiles)
    check_tree(pts, gpu_build(pts, depth=3, fourier_j=5), 5)

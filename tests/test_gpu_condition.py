"""The decision to re-solve a marker in double where an outer weight of its stencil is tiny: narrow weights, and home
cells beside much wider ones.

refined_fp64 is the number of markers whose cond_1(A) exceeds cond_max.  The single-precision estimate is a sum of
positive products of about 30 rounded factors, so it is held to a band of 0.1 % about the limit, and the limits are
placed inside the range that the markers span.
"""

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import run_gpu
from workloads import uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


def _setup(wide, K=1500):
    """z cells `wide` times as wide above the middle as below it (1: uniform)."""
    w = np.where(np.arange(16) < 8, 1.0, float(wide))
    f = np.concatenate([[0.0], np.cumsum(w)])
    faces = [uniform_faces(16), uniform_faces(16), f / f[-1] * 2 - 1]
    rng = np.random.default_rng(7)
    z = rng.uniform(faces[2][5], faces[2][11], K)
    z[: K // 3] = rng.uniform(faces[2][7], faces[2][8], K // 3)     # the last narrow cell
    x = np.stack([rng.uniform(-0.99, 0.99, K), rng.uniform(-0.99, 0.99, K), z]).astype(np.float32)
    return faces, (True, True, False), x, np.full(K, 1e-3, dtype=np.float32)


def _count(api, faces, periodic, x, area, eps, basis, cond_max):
    ctx = api.Context(faces, periodic, real="f32", eps=eps, basis=basis, cond_max=cond_max)
    return run_gpu(ctx, x, area, "exact")["status"]["refined_fp64"]


@pytest.mark.parametrize("wide,eps", [(1, 0.3), (1, 0.25), (8, 1.0), (10, 1.0), (10, 0.8)])
@pytest.mark.parametrize("basis", [4, 10])
def test_tiny_outer_weights(api, wide, eps, basis):
    faces, periodic, x, area = _setup(wide)
    _, cond = oracle.moment_matrix(oracle.Grid(faces, periodic), x.astype(np.float64), eps, basis=basis)
    limits = [1e6] + [float(np.quantile(cond, q)) for q in (0.05, 0.4, 0.8)]
    for lim in limits:
        if lim > 1e10:               # beyond what the double-precision inverse of the oracle resolves to 0.1 %
            continue
        n = _count(api, faces, periodic, x, area, eps, basis, lim)
        assert np.sum(cond > lim * 1.001) <= n <= np.sum(cond > lim * 0.999), (lim, n)

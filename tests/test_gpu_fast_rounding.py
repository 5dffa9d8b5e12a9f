"""Rounding error of the single-precision fast-MLS shape functions against the oracle's table blend in double.

A table row rounded once and blended with weights whose sum is off by a rounding or two has an rms error of about six
roundings of 2^-24 / sqrt(3) = 3.4e-8 in quadrature, 8.4e-8 of phi's norm; the product form must not exceed it.
"""

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import run_gpu, run_oracle
from workloads import tanh_faces, uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


@pytest.mark.parametrize("basis", [4, 10])
@pytest.mark.parametrize("axis", [None, 0, 2])
def test_rounding(api, axis, basis):
    faces = [uniform_faces(16), uniform_faces(16), uniform_faces(16)]
    if axis is not None:
        faces[axis] = np.round(tanh_faces(24, 1.2) * 2 ** 20) / 2 ** 20
    rng = np.random.default_rng(11)
    K = 4000
    x = np.empty((3, K))
    for d, f in enumerate(faces):
        i = rng.integers(2, len(f) - 3, K)
        u = (rng.integers(0, 8, K) + rng.uniform(1e-3, 1 - 1e-3, K)) / 8
        x[d] = f[i] + u * (f[i + 1] - f[i])
    x = x.astype(np.float32)
    periodic = (True, False, True)
    g = run_gpu(api.Context(faces, periodic, real="f32", basis=basis), x, np.full(K, 1e-3, np.float32), "fast")
    r = run_oracle(oracle.Grid(faces, periodic), x, np.full(K, 1e-3), "fast", basis=basis)
    assert np.linalg.norm(g["phi"] - r["phi"]) <= 8.4e-8 * np.linalg.norm(r["phi"])

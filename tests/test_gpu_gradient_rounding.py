"""Gradients away from the default weight, their rounding error on rough and smooth fields, and infinite field values.

Tolerances.  Normwise 1e-5 (single) and 1e-12 (double), as for the shape functions: about 30 roundings of O(1) terms,
plus a position's rounding against a face.  The rms error: a derivative is about 12 roundings deep, each with an rms
of 2^-24 / sqrt(3) = 3.4e-8, 1.2e-7 in quadrature, and the exponential adds its own: 1.5e-7 of the gradient's norm
whether the field varies from cell to cell or not.
"""

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import DEV, NP_DT, normwise
from workloads import tanh_faces, uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


def _gradient(api, faces, periodic, x, u, real, eps=1.0):
    K = x.shape[1]
    ctx = api.Context(faces, periodic, real=real, eps=eps)
    T = ctx.transfer(K)
    xt = torch.as_tensor(x, device=DEV)
    ctx.build_transfer(T, xt, torch.full((K,), 1e-3, dtype=xt.dtype, device=DEV))
    return ctx.interpolate_gradient(T, xt, torch.as_tensor(u, device=DEV)).double().cpu().numpy()


def _reference(faces, periodic, x, u, eps=1.0):
    grid = oracle.Grid(faces, periodic)
    x = x.astype(np.float64)
    return oracle.interpolate_gradient(oracle.shape_exact_gradient(grid, x, eps), oracle.support(grid, x),
                                       u.astype(np.float64))


def _markers(faces, K, real, seed):
    rng = np.random.default_rng(seed)
    return np.stack([rng.uniform(f[2], f[-3], K) for f in faces]).astype(NP_DT[real])


@pytest.mark.parametrize("real,tol", [("f64", 1e-12), ("f32", 1e-5)])
@pytest.mark.parametrize("kind,eps", [("uniform", 0.5), ("uniform", 3.0), ("tanh", 0.7), ("tanh", 2.0), ("narrow", 2.0),
                                      ("narrow", 3.0)])
def test_weights(api, kind, eps, real, tol):
    w = np.where(np.isin(np.arange(16), [3, 7, 11]), 1.0, 8.0)     # narrow cells between cells 8 times wider
    f = np.concatenate([[0.0], np.cumsum(w)])
    z = {"uniform": uniform_faces(32), "tanh": tanh_faces(24, 1.5), "narrow": f / f[-1] * 2 - 1}[kind]
    faces, periodic = [uniform_faces(16), uniform_faces(8), z], (True, True, False)
    x = _markers(faces, 1500, real, 41)
    u = np.random.default_rng(42).normal(size=(3, len(z) - 1, 8, 16)).astype(NP_DT[real])
    assert normwise(_gradient(api, faces, periodic, x, u, real, eps), _reference(faces, periodic, x, u, eps)) <= tol


@pytest.mark.parametrize("waves", [16, 2])
@pytest.mark.parametrize("stretch", [False, True])
def test_rounding(api, stretch, waves):
    """48^3, eight Fourier modes with up to `waves` periods in the box; faces that single precision holds, so that
    only the gradient's own rounding counts."""
    n = 48
    even = (np.arange(n + 1) - n // 2) / (n // 2 + 8.0)
    faces = [even, even, tanh_faces(n, 1.5).astype(np.float32).astype(np.float64) if stretch else even]
    periodic = (True, True, not stretch)
    rng = np.random.default_rng(5)
    Z, Y, X = np.meshgrid(*[0.5 * (f[1:] + f[:-1]) for f in faces[::-1]], indexing="ij")
    u = np.zeros((3, n, n, n))
    for c in range(3):
        for _ in range(8):
            k = rng.integers(-waves, waves + 1, 3) * 2 * np.pi / [f[-1] - f[0] for f in faces]
            u[c] += rng.normal() * np.sin(k[0] * X + k[1] * Y + k[2] * Z + rng.uniform(0, 2 * np.pi))
    u = u.astype(np.float32)
    x = _markers(faces, 20000, "f32", 6)
    ref = _reference(faces, periodic, x, u)
    err = np.linalg.norm(_gradient(api, faces, periodic, x, u, "f32") - ref) / np.linalg.norm(ref)
    assert err <= 1.5e-7, err


@pytest.mark.parametrize("real", ["f32", "f64"])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_values(api, real, bad):
    """One bad cell: markers that reach it get what the sum over the nodes gives, the others are untouched."""
    faces, periodic = [uniform_faces(16)] * 3, (True, True, True)
    x = _markers(faces, 4000, real, 8)
    x[:, :2000] = np.random.default_rng(10).uniform(-0.125, 0.25, (3, 2000))   # its home cell and the cells around
    u = np.random.default_rng(9).normal(size=(3, 16, 16, 16)).astype(NP_DT[real])
    clean = _gradient(api, faces, periodic, x, u, real)
    u[1, 8, 8, 8] = bad
    got = _gradient(api, faces, periodic, x, u, real)
    with np.errstate(invalid="ignore"):
        ref = _reference(faces, periodic, x, u)
    hit = ~np.isfinite(ref)
    assert 0 < hit.any(axis=(0, 1)).sum() < 4000 and not hit[[0, 2]].any()
    assert np.array_equal(got[~hit], clean[~hit])
    sure = hit & (np.abs(clean) < 1e30)
    same = np.isnan(ref) & np.isnan(got) | (ref == got)
    assert np.mean(same[sure]) > 0.999          # a weight within rounding of zero may take either sign

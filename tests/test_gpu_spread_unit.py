"""Rounding of the spread on well filled tiles, and the loops that only many markers or many tiles reach: chunks after
the first, zero and tiny chunks among others, several tiles per block, with and without 16-byte loads and reductions.

The reference is sum_l c_l phi_k F_l in double precision with the library's own phi and c.  The fixed-point unit is at
most 2^-22 of the largest |c F|; a run (up to four markers of a cell) rounds once, with an rms of unit / sqrt(12), and
the sum of a chunk is added to f in single precision (rms 2^-24 / sqrt(3) of the sum).  A cell's error therefore has
an rms of at most sqrt(runs / 12) unit + sqrt((adds + 4) / 3) 2^-24 times the sums' size, adds the number of such
additions.
"""

import numpy as np
import pytest
import torch

from gpu_helpers import DEV, gpu_transfer
from workloads import uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


def _build(api, n, x, cap, brick=(3, 3, 3), **kw):
    ctx = api.Context([uniform_faces(m) for m in n], (True, True, True), real="f32", brick_log2=brick, **kw)
    T = ctx.transfer(cap)
    M = x.shape[1]
    ctx.build_transfer(T, torch.as_tensor(x.astype(np.float32), device=DEV), torch.full((M,), 1e-3, device=DEV))
    return (ctx, T) + gpu_transfer(ctx, T)


def _spread(ctx, T, F, offset=0):
    """f from a field that starts `offset` floats behind an aligned address."""
    n = ctx.n
    buf = torch.zeros((3 * n[0] * n[1] * n[2] + offset,), device=DEV)
    f = buf[offset:].reshape(3, n[2], n[1], n[0])
    ctx.spread(T, torch.as_tensor(F.astype(np.float32), device=DEV), f)
    return f.double().cpu().numpy().reshape(3, -1)


def _reference(n, phi, c, home, F):
    F = F.astype(np.float32).astype(np.float64)
    i = [home % n[0], home // n[0] % n[1], home // (n[0] * n[1])]
    N = n[0] * n[1] * n[2]
    ref, size, terms = np.zeros((3, N)), np.zeros((3, N)), np.zeros(N)
    for k in range(27):
        z, y, x = ((i[2] + k // 9 - 1) % n[2], (i[1] + k // 3 % 3 - 1) % n[1], (i[0] + k % 3 - 1) % n[0])
        cell = (z * n[1] + y) * n[0] + x
        terms += np.bincount(cell, minlength=N)
        for q in range(3):
            t = c * phi[:, k] * F[q]
            ref[q] += np.bincount(cell, weights=t, minlength=N)
            size[q] += np.bincount(cell, weights=np.abs(t), minlength=N)
    return ref, size, terms


@pytest.mark.parametrize("per_tile", [100, 250, 500, 4096])
@pytest.mark.parametrize("value", [1.0, 1.9])
def test_equal_forces(api, per_tile, value):
    """`per_tile` markers in each of 18 tiles, forces of one size and either sign: the unit's error stands out, since
    the sums in f stay small (three times the root of the sum of squares bounds them with few exceptions)."""
    n = (24, 24, 16)
    rng = np.random.default_rng(per_tile)
    M = 18 * per_tile
    ctx, T, phi, c, home = _build(api, n, rng.uniform(-1, 1, (3, M)), M)
    F = value * rng.choice([-1.0, 1.0], (3, M))
    ref, _, terms = _reference(n, phi, c, home, F)
    square = _reference(n, phi * phi, c * c, home, F * F)[0]
    unit = 2.0 ** -22 * np.max(np.abs(c * F))
    adds = 8 + per_tile / 256                         # up to eight tiles or shares of one, and their chunks
    sigma = np.sqrt((terms / 4 + 8) / 12) * unit + np.sqrt((adds + 4) / 3) * 2.0 ** -24 * 3 * np.sqrt(square)
    err = _spread(ctx, T, F) - ref
    at = terms > 0
    assert np.sqrt(np.mean((err[:, at] / sigma[:, at]) ** 2)) <= 1.0


@pytest.mark.parametrize("basis,eps", [(4, 0.5), (10, 1.0)])
def test_large_shape_functions(api, basis, eps):
    """|phi| up to 0.9 and full chunks: terms above the chunk's limit are added directly, none is lost."""
    n, M = (16, 16, 16), 9000
    rng = np.random.default_rng(3)
    x = rng.uniform(-0.45, -0.05, (3, M))
    x[:, ::3] = (np.floor(x[:, ::3] * 8) + 0.5) / 8 + rng.uniform(-0.002, 0.002, x[:, ::3].shape)   # cell centres
    ctx, T, phi, c, home = _build(api, n, x, M, eps=eps, basis=basis)
    assert np.max(np.abs(phi)) > 0.5
    F = rng.normal(size=(3, M))
    ref, size, terms = _reference(n, phi, c, home, F)
    bound = terms * 2.0 ** -21 * np.max(np.abs(c * F)) + (5 + terms) * 2.0 ** -24 * size
    assert np.all(np.abs(_spread(ctx, T, F) - ref) <= bound)


@pytest.mark.parametrize("nx,extra,offset", [(16, 0, 0), (16, 1, 0), (18, 0, 0), (16, 0, 1), (18, 1, 1)])
def test_many_chunks(api, nx, extra, offset):
    """More than 8 x 512 markers in one tile, with stretches of zero and of tiny forces in the stored order."""
    n, M = (nx, 16, 16), 12001
    rng = np.random.default_rng(nx + extra)
    x = rng.uniform(-0.45, -0.05, (3, M))
    ctx, T, phi, c, home = _build(api, n, x, M + extra)
    perm = ctx.view(T)["perm"].cpu().numpy()
    F = rng.normal(size=(3, M))
    F[:, perm[1000:3200]] = 0.0
    F[:, perm[5000:7100]] *= 1e-12
    ref, size, terms = _reference(n, phi, c, home, F)
    bound = terms * 2.0 ** -22 * np.max(np.abs(c * F)) + (5 + M / 256) * 2.0 ** -24 * size
    assert np.all(np.abs(_spread(ctx, T, F, offset) - ref) <= bound)


@pytest.mark.parametrize("nx", [66, 64])
@pytest.mark.parametrize("extra", [0, 1])
def test_more_tiles_than_blocks(api, nx, extra):
    """Up to 33 792 tiles of 2 x 2 x 2 cells: every resident block walks a range of them."""
    n, M = (nx, 64, 64), 80000
    rng = np.random.default_rng(nx + extra)
    x = rng.uniform(-0.999, 0.999, (3, M))
    x[:, :3000] = 0.3 + rng.uniform(0, 0.02, (3, 3000))            # one crowded tile among them
    ctx, T, phi, c, home = _build(api, n, x, M + extra, brick=(1, 1, 1))
    F = rng.normal(size=(3, M))
    ref, size, terms = _reference(n, phi, c, home, F)
    bound = terms * 2.0 ** -22 * np.max(np.abs(c * F)) + 40 * 2.0 ** -24 * size
    assert np.all(np.abs(_spread(ctx, T, F) - ref) <= bound)

"""Collision flags by blocks and by warps: tiles of 2^11 and more cells, crowded tiles (thousands of markers in one),
few tiles and many, equal to the oracle's integers."""

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import DEV
from oracle.collision import collision_cells, collision_flags
from workloads import uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


@pytest.mark.parametrize("n,M,crowd,brick", [
    ((64, 64, 64), 20000, 0, (4, 4, 3)),           # tiles of 2^11 cells: blocks only
    ((64, 64, 64), 20000, 6000, (5, 4, 4)),        # 2^13 cells, one crowded
    ((32, 32, 32), 9000, 6000, (3, 3, 3)),         # few tiles, thousands of markers in one: blocks
    ((32, 32, 32), 3, 0, (3, 3, 3)),
    ((66, 64, 64), 50000, 0, (1, 1, 1)),           # tens of thousands of tiles: warps
    ((66, 64, 64), 50000, 6000, (1, 1, 2)),        # and a crowded one among them
    ((48, 64, 80), 60000, 700, (2, 2, 2)),         # about as many tiles as blocks
])
def test_forms(api, n, M, crowd, brick):
    rng = np.random.default_rng(M + crowd)
    faces = [uniform_faces(m) for m in n]
    grid = oracle.Grid(faces, (True, True, False))
    x = rng.uniform(-0.999, 0.999, (3, M))
    x[:, :crowd] = 0.31 + rng.uniform(0, 2.0 / n[0], (3, crowd))
    x = np.ascontiguousarray(x[:, rng.permutation(M)], dtype=np.float32)
    body = rng.integers(0, 4, M).astype(np.int32)
    ctx = api.Context(faces, (True, True, False), real="f32", brick_log2=brick)
    T = ctx.transfer(M)
    ctx.build_transfer(T, torch.as_tensor(x, device=DEV), torch.full((M,), 1e-3, device=DEV))
    coll = torch.zeros(n[::-1], dtype=torch.int32, device=DEV)
    count = torch.zeros(1, dtype=torch.int64, device=DEV)
    flag = ctx.collisions(T, torch.as_tensor(body, device=DEV), coll=coll, count=count).cpu().numpy()
    home, ok = oracle.locate(grid, x.astype(np.float64))
    want = collision_flags(home, ok, body, grid.n)
    keys, state = collision_cells(home, ok, body, grid.n)
    assert np.array_equal(flag, want) and int(count.item()) == int(want.sum())
    got = coll.cpu().numpy().ravel()
    assert np.array_equal(np.nonzero(got)[0], keys) and np.array_equal(got[keys], state)

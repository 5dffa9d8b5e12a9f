"""Interpolation and direct forcing by tiles: tile shapes, x extents that are a multiple of 4, even or odd and that end
inside a tile, walls, fields off a 16-byte boundary, bfloat16, capacities off a multiple of 4, crowded tiles shared by
several blocks, tiles too large for one pass, u and f in one buffer, infinite velocities.

The references are double-precision sums with the library's own phi, c and F.  U: 27 fused multiply-adds, 28 x 2^-24
sum |phi u|.  f: the fixed-point unit is at most 2^-22 of the largest |c F| and each term rounds once (half a unit)
after one rounding of its own; f is accumulated in single precision once per chunk, (6 + chunks) 2^-24 sum |c phi F|.
bfloat16 fields round every addition to f: 2^-8 of the sum's largest partial value, bounded by 2^-8 adds sum |c phi F|.
"""

import numpy as np
import pytest
import torch

from gpu_helpers import DEV, TORCH_DT, gpu_transfer
from workloads import tanh_faces, uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


def _setup(api, nx, M, cap, brick, periodic, field, seed, ny=12, nz=20):
    n = (nx, ny, nz)
    faces = [uniform_faces(nx), uniform_faces(ny), tanh_faces(nz, 1.5)]
    rng = np.random.default_rng(seed)
    x = np.stack([rng.uniform(f[0], f[-1], M) for f in faces]) * 0.999          # some in wall cells: dropped
    x[:, M // 2:] = x[:, :1] * 0.8 + rng.uniform(-0.05, 0.05, (3, M - M // 2))   # half of them crowd a few cells
    ctx = api.Context(faces, (periodic, True, False), real="f32", field=field, brick_log2=brick)
    T = ctx.transfer(cap)
    ctx.build_transfer(T, torch.as_tensor(x.astype(np.float32), device=DEV), torch.full((M,), 1e-3, device=DEV))
    return ctx, T, n, rng, gpu_transfer(ctx, T)


def _field(n, field, offset, rng=None):
    """A field that starts `offset` elements behind an aligned address, random or zero."""
    N = 3 * n[0] * n[1] * n[2]
    buf = torch.zeros(N + offset, dtype=TORCH_DT[field], device=DEV)
    if rng is not None:
        buf[offset:] = torch.as_tensor(rng.normal(size=N), device=DEV).to(buf.dtype)
    return buf[offset:].reshape(3, n[2], n[1], n[0])


def _cells(n, home):
    ok = home >= 0
    h = np.where(ok, home, 0)
    i = [h % n[0], h // n[0] % n[1], h // (n[0] * n[1])]
    for k in range(27):
        z, y, x = i[2] + k // 9 - 1, (i[1] + k // 3 % 3 - 1) % n[1], (i[0] + k % 3 - 1) % n[0]
        yield k, ok, (np.clip(z, 0, n[2] - 1) * n[1] + y) * n[0] + x


def _check(n, tr, u, Vb, dt, U, F, f, field):
    phi, c, home = tr
    u = u.double().cpu().numpy().reshape(3, -1)
    U, F = U.double().cpu().numpy(), F.double().cpu().numpy()
    M = phi.shape[0]
    ref, size = np.zeros((3, M)), np.zeros((3, M))
    fr, fs, terms = (np.zeros((3, u.shape[1])) for _ in range(3))
    for k, ok, cell in _cells(n, home):
        ref += phi[:, k] * u[:, cell] * ok
        size += np.abs(phi[:, k] * u[:, cell]) * ok
        for q in range(3):
            t = (c * phi[:, k] * F[q])[ok]
            fr[q] += np.bincount(cell[ok], weights=t, minlength=u.shape[1])
            fs[q] += np.bincount(cell[ok], weights=np.abs(t), minlength=u.shape[1])
            terms[q] += np.bincount(cell[ok], minlength=u.shape[1])
    assert np.all(np.abs(U - ref) <= 28 * 2.0 ** -24 * size)
    want = np.where(home >= 0, (Vb.double().cpu().numpy() - U) / dt, 0.0)
    assert np.all(np.abs(F - want) <= 4 * 2.0 ** -24 * np.abs(want) + 1e-30)
    err = np.abs(f.double().cpu().numpy().reshape(3, -1) - fr)
    top = np.max(np.abs(c * F), axis=1)[:, None]
    adds = 8 + M / 128 if field == "f32" else terms + 8
    assert np.all(err <= terms * 2.0 ** -23 * top + (6 + adds) * (2.0 ** -24 if field == "f32" else 2.0 ** -8) * fs)


@pytest.mark.parametrize("brick", [(3, 3, 3), (2, 3, 1), (1, 2, 3), (4, 4, 3), (5, 1, 2), (5, 4, 4)])
@pytest.mark.parametrize("nx,periodic", [(20, True), (18, True), (17, True), (16, False), (4, True)])
@pytest.mark.parametrize("M,cap,field,offset", [(3, 3, "f32", 0), (900, 901, "f32", 1), (5000, 5000, "f32", 0),
                                                (900, 901, "bf16", 0), (900, 900, "bf16", 1)])
def test_direct_forcing(api, M, cap, field, offset, nx, periodic, brick):
    ctx, T, n, rng, tr = _setup(api, nx, M, cap, brick, periodic, field, M + nx)
    u, f = _field(n, field, offset, rng), _field(n, field, offset)
    Vb = torch.as_tensor(rng.normal(size=(3, M)).astype(np.float32), device=DEV)
    U = torch.full((3, M), 7.0, device=DEV)
    F, _ = ctx.direct_forcing(T, u, Vb, 1e-2, f, U=U)
    _check(n, tr, u, Vb, 1e-2, U, F, f, field)
    only = ctx.interpolate(T, u)
    assert torch.equal(only, U)
    f2 = _field(n, field, offset)
    F2, none = ctx.direct_forcing(T, u, Vb, 1e-2, f2)
    assert none is None and torch.equal(F2, F)


def test_many_tiles(api):
    """More tiles than blocks: every block takes several."""
    ctx, T, n, rng, tr = _setup(api, 66, 60000, 60001, (1, 1, 1), True, "f32", 3, ny=48, nz=48)
    u, f = _field(n, "f32", 0, rng), _field(n, "f32", 0)
    Vb = torch.as_tensor(rng.normal(size=(3, 60000)).astype(np.float32), device=DEV)
    U = torch.empty((3, 60000), device=DEV)
    F, _ = ctx.direct_forcing(T, u, Vb, 1e-2, f, U=U)
    _check(n, tr, u, Vb, 1e-2, U, F, f, "f32")


def test_field_shared_with_f(api):
    """f accumulated on top of u: the forces come from u as it was."""
    ctx, T, n, rng, tr = _setup(api, 16, 2000, 2000, (3, 3, 3), True, "f32", 4)
    u = _field(n, "f32", 0, rng)
    Vb = torch.as_tensor(rng.normal(size=(3, 2000)).astype(np.float32), device=DEV)
    f = _field(n, "f32", 0)
    F, _ = ctx.direct_forcing(T, u, Vb, 1e-2, f)
    both = u.clone()
    F2, _ = ctx.direct_forcing(T, both, Vb, 1e-2, both)
    assert torch.equal(F, F2)
    assert float((both - u - f).abs().max()) <= 2.0 ** -18 * float(f.abs().max())


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_velocity(api, bad):
    ctx, T, n, rng, (phi, c, home) = _setup(api, 20, 1500, 1500, (3, 3, 3), True, "f32", 5)
    u = _field(n, "f32", 0, rng)
    l = int(np.nonzero(home >= 0)[0][0])
    u.view(3, -1)[1, int(home[l])] = bad
    f = _field(n, "f32", 0)
    F, _ = ctx.direct_forcing(T, u, torch.zeros((3, 1500), device=DEV), 1e-2, f)
    F = F.double().cpu().numpy()
    assert np.isfinite(F[[0, 2]]).all() and not np.isfinite(F[1, l])
    hit = np.zeros((3, n[0] * n[1] * n[2]), dtype=bool)
    for k, ok, cell in _cells(n, home):
        for q in range(3):
            hit[q, cell[ok & ~np.isfinite(F[q])]] = True
    got = f.double().cpu().numpy().reshape(3, -1)
    assert not np.isfinite(got[hit]).any() and np.isfinite(got[~hit]).all()

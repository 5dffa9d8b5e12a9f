"""Fast-MLS builds without the table: device memory of a first build, and the table made where it is asked for."""

import numpy as np
import pytest
import torch

from gpu_helpers import DEV, gpu_transfer
from workloads import tanh_faces, uniform_faces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1805_01113_gb300 import api as _api
    torch.cuda.set_device(0)
    return _api


def _build(ctx, x, area):
    T = ctx.transfer(x.shape[1])
    ctx.build_transfer(T, x, area, "fast")
    torch.cuda.synchronize()
    return torch.as_tensor(gpu_transfer(ctx, T)[0])        # in the caller's order: the stored one may differ


def _inputs(K=500):
    rng = np.random.default_rng(1)
    x = torch.as_tensor(rng.uniform(-0.8, 0.8, (3, K)).astype(np.float32), device=DEV)
    return x, torch.full((K,), 1e-3, device=DEV)


def test_first_build_needs_no_table(api):
    """512 classes of 33^3 rows are 2 GB; a build takes the factors (0.5 MB) and its transfer."""
    ctx = api.Context([uniform_faces(16), uniform_faces(16), tanh_faces(512, 1.5)], (True, True, False), n_sub=33)
    x, area = _inputs()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    _build(ctx, x, area)
    assert before - torch.cuda.mem_get_info()[0] < 64 << 20


def test_table_on_request(api, tmp_path):
    faces, periodic = [uniform_faces(16), uniform_faces(16), tanh_faces(24, 1.5)], (True, True, False)
    x, area = _inputs()
    built, asked = api.Context(faces, periodic), api.Context(faces, periodic)
    table = asked.fast_table().cpu()
    phi = _build(built, x, area)
    assert torch.equal(_build(asked, x, area), phi)
    built.save(tmp_path / "built")                     # as after mls_fast_table
    asked.save(tmp_path / "asked")
    assert (tmp_path / "built").read_bytes() == (tmp_path / "asked").read_bytes()
    loaded = api.Context(faces, periodic)
    loaded.load(tmp_path / "built")
    loaded.timing(True)
    assert torch.equal(loaded.fast_table().cpu(), table) and torch.equal(_build(loaded, x, area), phi)
    assert not {"fast_table", "fast_axes"} & set(loaded.read_timing())
    built.load(tmp_path / "asked")                     # over existing state
    assert torch.equal(built.fast_table().cpu(), table) and torch.equal(_build(built, x, area), phi)

"""The two-value plane walks by 32-bit offset, and the static one by address.

Frame pairs and Thomson B pairs lie in the library's own buffers; the walks
step addresses where every unit of the buffers lies between two multiples of
2^32, and go by offset otherwise.  Pair buffers of more than 2^32 bytes in
units that do not divide 2^32, and B buffers less than 2^21 bytes short of
2^32 (large allocations start on multiples of 2^21), cross one wherever they
are.  Both forms visit the per-ray walk's segments in its order (Section
3.3.1, Eq. lo; Section 3.3.3 for frames): equal bit for bit."""

import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()
    yield
    torch.cuda.empty_cache()


@pytest.fixture(scope="module")
def T():
    import paper_1103_5904_gb300 as T
    return T


def _views(n_img, npx, fov=3.2):
    """Views of every layout: along x, along y, rolled by 90 degrees, tilted."""
    k = np.arange(n_img)
    p = synth.pointing_table(30.0 + 70.0 * k, np.where(k % 4 == 3, 40.0, 1.0),
                             215.0, npx, npx, fov)
    p[k % 4 == 2, 3] = np.pi / 2
    return p


def _project(T, plane_sync, x, g, p, npx, **kw):
    ctx = T.Context()
    ctx.set_option(T.tomo.TOMO_OPT_PLANE_SYNC, plane_sync)
    y = T.tomo_project(x, g, p, npx, npx, ctx=ctx, **kw)
    ctx.close()
    return y


@pytest.mark.parametrize("dtype,frames", [(torch.float32, 270),
                                          (torch.bfloat16, 540)])
def test_frame_pairs_by_offset(T, dtype, frames):
    nx, ny, nz, npx = 127, 129, 131, 24
    n, size = nx * ny * nz, 8 if dtype == torch.float32 else 4
    assert n % 2 and size * n * (frames - 1) > 1 << 32
    g = synth.cube_geom(nx, 1.5, ny, nz)
    p = _views(2 * (frames - 1), npx)
    p[:, 11] = (np.arange(len(p)) + 0.5) / 2  # every pair of frames
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    x = torch.rand((frames, nz, ny, nx), generator=gen, device="cuda").to(dtype)
    got = _project(T, 3, x, g, p, npx, n_frames=frames)
    assert torch.equal(got, _project(T, 0, x, g, p, npx, n_frames=frames))
    assert (got > 0).any()


def test_thomson_b_by_offset(T):
    nx, ny, nz, npx = 812, 813, 813, 64
    assert 0 <= (1 << 32) - 8 * nx * ny * nz < 1 << 21
    g = synth.cube_geom(nx, 1.5, ny, nz)
    p = _views(4, npx)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    x = torch.rand((nz, ny, nx), generator=gen, device="cuda")
    kw = {"kind": "B", "limb_u": 0.6}
    got = _project(T, 3, x, g, p, npx, **kw)
    assert torch.equal(got, _project(T, 0, x, g, p, npx, **kw))
    assert (got != 0).any()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_static_by_address(T, dtype):
    n, npx = 40, 48
    g, p = synth.cube_geom(n, 1.5), _views(4, npx)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x = torch.rand((n, n, n), generator=gen, device="cuda").to(dtype)
    last = x.data_ptr() + x.numel() * x.element_size() - 1
    assert x.data_ptr() >> 32 == last >> 32
    got = _project(T, 3, x, g, p, npx)
    assert torch.equal(got, _project(T, 0, x, g, p, npx))

"""The gathering plane walks by address and by offset.

A walk whose buffers (the cube and its layout copies) lie between two
multiples of 2^32 bytes steps the low half of each voxel's address; any other
buffer is walked by 32-bit offsets from its base.  Both visit the same
segments in the same order (Section 3.3.1, Eq. lo), so a cube placed across a
multiple of 2^32 gives the same images, bit for bit, as the same cube placed
anywhere else, whatever the layout its images walk and its storage type."""

import numpy as np
import pytest
import torch

import synth
from oracle import siddon
from tests.gpu_util import assert_close, require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.fixture(scope="module")
def T():
    import paper_1103_5904_gb300 as T
    return T


@pytest.fixture(scope="module")
def pool():
    """A byte buffer of more than 2^32 bytes: it holds a multiple of 2^32."""
    p = torch.empty((1 << 32) + (64 << 20), dtype=torch.uint8, device="cuda")
    yield p
    del p
    torch.cuda.empty_cache()


def _across(pool, x, before):
    """A copy of x in the pool whose first `before` bytes lie below the
    multiple of 2^32 that the pool holds."""
    n = x.numel() * x.element_size()
    base = pool.data_ptr()
    edge = (base + (32 << 20) + (1 << 32) - 1) >> 32 << 32
    at = edge - before - base
    assert at >= 0 and at + n <= pool.numel()
    y = pool[at:at + n].view(x.dtype).view(x.shape)
    y.copy_(x)
    assert (y.data_ptr() >> 32) != ((y.data_ptr() + n - 1) >> 32)
    return y


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("lat", [0.0, 12.0], ids=["counted", "every slab"])
def test_cube_across_a_multiple_of_2_32(T, pool, dtype, lat):
    g = {"nx": 37, "ny": 41, "nz": 33, "x0": -1.5, "y0": -1.45, "z0": -1.4,
         "dx": 3.0 / 37, "dy": 2.9 / 41, "dz": 2.8 / 33}
    # rows along x, y and (rolled) z: every layout, the native one included
    ptg = synth.pointing_table([3.0, 88.0, 40.0, 200.0], lat, 215.0, 45, 39, 3.3)
    ptg[2, 3] = np.pi / 2
    rng = np.random.default_rng(3)
    x = to_dev(rng.random((33, 41, 37)).astype(np.float32)).to(dtype)
    ctx = T.Context()
    ctx.set_option(T.tomo.TOMO_OPT_PLANE_SYNC, 3)  # every image by plane
    want = T.tomo_project(x, g, ptg, 45, 39, ctx=ctx)
    n = x.numel() * x.element_size()
    for before in (4, n // 8 * 4, n - 4):
        got = T.tomo_project(_across(pool, x, before), g, ptg, 45, 39, ctx=ctx)
        assert torch.equal(got, want), before
    ctx.close()
    assert_close(want.cpu().numpy(),
                 siddon.project(g, x.float().cpu().numpy(), ptg, 45, 39),
                 "P near buffers")

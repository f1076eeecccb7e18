"""Which forward the built-in walk rules choose.

A pixel pitch just below the plane forward's threshold must cost what it
cost without the plane walk: one per-ray launch, no layout copy and no launch
that finds nothing to do.  Tilted views with pixels 0.5 to 0.75 voxel apart
take the plane forward only on large cubes and only where it takes every
image; for one value per voxel, only where the rows of voxels are whole
128-byte lines (elsewhere it measured up to 25 % slower).  The walk is a matter of speed only (Section
3.3.1, Eq. lo)."""

import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.fixture(scope="module")
def T():
    import paper_1103_5904_gb300 as T
    return T


def _views(n, npx, pitch, lat=7.0, n_img=6):
    """Tilted views with pixels `pitch` voxels apart at Sun centre."""
    p = synth.pointing_table(np.arange(n_img) * 30.0 + 7.3, lat, 215.0, npx,
                             npx, 3.0)
    p[:, 4:6] = np.arctan(pitch * (3.0 / n) / 215.0)
    return p


@pytest.mark.parametrize("kind", ["static", "frames"])
@pytest.mark.parametrize("below", [0.999, 0.95])
def test_below_the_threshold_one_launch(T, kind, below):
    n, npx, frames = 33, 40, 3 if kind == "frames" else 1
    g, p = synth.cube_geom(n, 1.5), _views(n, npx, 0.6)
    p[:, 11] = np.linspace(0.0, frames - 1.0, len(p))
    ctx = T.Context()
    T.tomo_set_plane_rules({"fwd_min_pitch": 0.6 / below, "fwd_max_ratio": 0.0},
                           ctx=ctx)
    shape = (n,) * 3 if frames == 1 else (frames,) + (n,) * 3
    x = to_dev(np.random.default_rng(3).random(shape).astype(np.float32))
    T.tomo_project(x, g, p, npx, npx, n_frames=frames, ctx=ctx)
    ctx.profile(reset=True)
    got = T.tomo_project(x, g, p, npx, npx, n_frames=frames, ctx=ctx)
    count = ctx.profile(reset=True)
    assert not ((T.tomo_walk_plan(len(p), ctx=ctx) & 2) != 0).any()
    assert count["forward"][0] == 1 and count["layout"][0] == 0, count
    ctx.set_option(T.tomo.TOMO_OPT_PLANE_SYNC, 0)
    assert torch.equal(got, T.tomo_project(x, g, p, npx, npx, n_frames=frames,
                                           ctx=ctx))
    ctx.close()


@pytest.mark.parametrize("shape,dtype,frames,kind,plane", [
    ((128, 128, 128), "f32", 1, "emission", True),
    ((128, 128, 128), "bf16", 1, "emission", True),
    ((101, 101, 101), "f32", 1, "emission", False),  # below 2^20 voxels
    ((104, 104, 104), "f32", 1, "emission", False),  # 416-byte rows
    ((127, 128, 128), "f32", 1, "emission", False),
    ((160, 96, 96), "f32", 1, "emission", True),     # 640-byte rows
    ((160, 96, 96), "bf16", 1, "emission", False),   # 320-byte rows
    ((160, 96, 96), "bf16", 1, "pB", True),          # walks floats
    ((104, 104, 104), "f32", 2, "emission", True),   # frame pairs
    ((104, 104, 104), "f32", 1, "B", True),          # one walk, two values
])
def test_default_forward(T, shape, dtype, frames, kind, plane):
    nx, ny, nz = shape
    npx = 16
    g, p = synth.cube_geom(nx, 1.5, ny, nz), _views(nx, npx, 0.6, n_img=2)
    p[:, 1] = np.deg2rad([97.0, 263.0])  # along y: image rows along x
    x = torch.ones(((frames,) if frames > 1 else ()) + (nz, ny, nx),
                   device="cuda")
    x = x.to(torch.bfloat16) if dtype == "bf16" else x
    ctx = T.Context()
    for pitch, want in ((0.6, plane), (0.45, False), (0.8, True)):
        p[:, 4:6] = np.arctan(pitch * (3.0 / nx) / 215.0)
        T.tomo_project(x, g, p, npx, npx, n_frames=frames, kind=kind, ctx=ctx)
        code = T.tomo_walk_plan(len(p), ctx=ctx)
        assert (((code & 2) != 0) == want).all(), (pitch, code)
    # one image below 0.5 voxel: each is held to 0.75 voxel, but where one
    # launch walks both kinds of image
    p[0, 4:6] = np.arctan(0.45 * (3.0 / nx) / 215.0)
    for pitch, want in ((0.6, kind == "B"), (0.8, True)):
        p[1, 4:6] = np.arctan(pitch * (3.0 / nx) / 215.0)
        T.tomo_project(x, g, p, npx, npx, n_frames=frames, kind=kind, ctx=ctx)
        code = T.tomo_walk_plan(len(p), ctx=ctx)
        assert ((code & 2) != 0).tolist() == [False, want], (pitch, code)
    ctx.close()


@pytest.mark.parametrize("bucket", [False, True], ids=["context", "bucket"])
def test_other_rules_keep_the_default_forward(T, bucket):
    """Setting one rule leaves the others at the built-in defaults of each
    cube, for the context as for a size bucket; setting all of them does not."""
    npx, ctx = 16, T.Context()
    for n, plane in ((128, True), (104, False)):
        g, p = synth.cube_geom(n, 1.5), _views(n, npx, 0.6, n_img=2)
        x = torch.ones((n,) * 3, device="cuda")

        def forward(rules):
            at = (g, npx, npx, 2) if bucket else ()
            T.tomo_set_plane_rules(rules, *at, ctx=ctx)
            T.tomo_project(x, g, p, npx, npx, ctx=ctx)
            code = T.tomo_walk_plan(len(p), ctx=ctx)
            assert ((code & 2) != 0).all() or not ((code & 2) != 0).any()
            return bool(code[0] & 2), bool(code[0] & 4)

        assert forward(None) == (plane, True)
        assert forward({"general_ratio": 1e30}) == (plane, False)
        assert forward({"fwd_group": 8.0}) == (plane, True)
        assert forward({"fwd_min_pitch": 0.55}) == (True, True)
        every = {"min_pitch": 0.16, "fwd_min_pitch": 0.75, "fwd_max_ratio": 0.02,
                 "general_ratio": 0.035, "fwd_group": 0.0, "adj_group": 0.0}
        assert forward(every) == (False, True)
        assert forward(None) == (plane, True)
    for bad in ({"min_pitch": -1.0}, {"general_ratio": float("nan")}):
        with pytest.raises(T.TomoError):
            T.tomo_set_plane_rules(bad, ctx=ctx)
    ctx.close()


def test_transpose_keeps_the_hints_of_the_forward(T):
    """A transpose between two forwards of a bf16 cube whose type decides the
    forward (320-byte rows) rebuilds nothing."""
    npx, ctx = 16, T.Context()
    g, p = synth.cube_geom(160, 1.5, 96, 96), _views(160, npx, 0.6, n_img=2)
    p[:, 1] = np.deg2rad([97.0, 263.0])  # along y: image rows along x
    x = torch.ones((96, 96, 160), device="cuda", dtype=torch.bfloat16)
    y = T.tomo_project(x, g, p, npx, npx, ctx=ctx)
    code = T.tomo_walk_plan(len(p), ctx=ctx)
    ctx.profile(reset=True)
    T.tomo_backproject(y, g, p, ctx=ctx)
    T.tomo_project(x, g, p, npx, npx, ctx=ctx)
    assert ctx.profile(reset=True)["setup"][0] == 0
    assert (T.tomo_walk_plan(len(p), ctx=ctx) == code).all()
    T.tomo_project(x.float(), g, p, npx, npx, ctx=ctx)
    assert ctx.profile(reset=True)["setup"][0] == 1  # the hints alone
    ctx.close()

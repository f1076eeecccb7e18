"""Which forward a stack takes where no image takes the plane walk.

A pixel pitch just below the plane forward's threshold must cost what it
cost without the plane walk: one per-ray launch, no layout copy and no launch
that finds nothing to do (the walk is a matter of speed only: Section 3.3.1,
Eq. lo)."""

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

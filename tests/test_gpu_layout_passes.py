"""The layout passes that a geometry does not need are not launched.

Which layouts of the cube the images of a geometry walk in is decided on the
device; the host evaluates the same rule with a margin and launches the copy,
zero and combine passes only of layouts that some image may use, and the
per-ray forward only when some image may need it.  Geometries on and around
the rule's ties (two axes equally steep, two lateral axes equally good, pixel
pitch and direction ratio on a threshold) and one-layout stacks must give the
per-ray walk's images bit for bit and its transpose up to the order of float
additions (Section 3.3.1, Eq. lo)."""

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


N, NPX = 33, 40


def _views(name):
    eps = 1e-12
    lon, lat, roll = {
        "one layout": ([2.0, -3.0, 178.0], [0.0, 0.0, 0.5], 0.0),
        "steepest axis tied": ([45.0, 45.0 + eps, 135.0 - eps, 225.0], 0.0, 0.0),
        "lateral axis tied": ([0.0, 90.0, 180.0, 10.0], 0.0, 45.0),
        "z tied": ([10.0, 100.0, 45.0], [45.0, 45.0 + eps, 35.264389682754654], 0.0),
        "all layouts": ([5.0, 95.0, 40.0], [0.0, 3.0, 10.0], [0.0, 0.0, 90.0]),
    }[name]
    lon = np.asarray(lon)
    p = synth.pointing_table(lon, lat, 215.0, NPX, NPX, 3.4)
    p[:, 3] = np.deg2rad(roll)
    return p


@pytest.mark.parametrize("name", ["one layout", "steepest axis tied",
                                  "lateral axis tied", "z tied", "all layouts"])
@pytest.mark.parametrize("rules", ["defaults", "on the thresholds"])
def test_layout_passes(T, name, rules):
    g = synth.cube_geom(N, 1.5)
    p = _views(name)
    rng = np.random.default_rng(9)
    x = to_dev(rng.random((N, N, N)).astype(np.float32))
    y = to_dev(rng.random((len(p), NPX, NPX)).astype(np.float32))
    ctx, ray = T.Context(), T.Context()
    ray.set_option(T.tomo.TOMO_OPT_PLANE_SYNC, 0)
    if rules != "defaults":
        pitch = float(p[0, 0] * abs(np.tan(p[0, 4])) / g["dx"])
        T.tomo_set_plane_rules({"min_pitch": pitch, "fwd_min_pitch": pitch,
                                "fwd_max_ratio": 0.0}, ctx=ctx)
    want = T.tomo_project(x, g, p, NPX, NPX, ctx=ray)
    want_t = T.tomo_backproject(y, g, p, ctx=ray)
    # a context's first call and one after another geometry used its buffers
    for k in range(2):
        assert torch.equal(T.tomo_project(x, g, p, NPX, NPX, ctx=ctx), want)
        # sums of at most 4 x 12 terms per voxel in another order: 1e-5 is far
        # above their rounding and far below a missing or stale term
        torch.testing.assert_close(T.tomo_backproject(y, g, p, ctx=ctx), want_t,
                                   rtol=1e-5, atol=1e-6 * float(want_t.max()))
        other = _views("all layouts")
        yo = to_dev(rng.random((len(other), NPX, NPX)).astype(np.float32))
        T.tomo_backproject(yo, g, other, ctx=ctx)
        T.tomo_project(x, g, other, NPX, NPX, ctx=ctx)
    ctx.close()
    ray.close()

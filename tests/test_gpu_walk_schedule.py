"""The launched passes are those that the device's walk choice needs.

Per image the device chooses major and lateral axis (the layout), plane or
per-ray walk and forward; the host launches the copy, zero and combine passes
of the layouts in use and the per-ray forward only where some image takes it.
Over random stacks (views anywhere, rolls, pixel pitches on both sides of the
thresholds, images of different layouts that do and do not take the plane
forward) the counts must be those of ``tomo_walk_plan``; with axes or
thresholds tied a pass may be launched in vain, never left out.  Images must
be the per-ray walk's bit for bit and transposes equal up to the order of
float additions of non-negative terms (at most a few dozen per voxel: 1e-5
is far above it, a missing or stale term far above 1e-5), for the static
model, frame pairs and Thomson B, also after another geometry used the
buffers."""

import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import require_gpu, to_dev

pytestmark = pytest.mark.gpu

N, NPX, FRAMES = 17, 23, 3
KINDS = {"static": (1, "emission"), "frames": (FRAMES, "emission"),
         "B": (1, "B")}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.fixture(scope="module")
def T():
    import paper_1103_5904_gb300 as T
    return T


def _stack(rng, tied):
    n = int(rng.integers(1, 5))
    if tied:
        lon = rng.choice([0.0, 45.0, 90.0, 135.0, 200.0], n)
        lat = rng.choice([0.0, 45.0, 35.264389682754654], n)
        roll = rng.choice([0.0, 45.0, 90.0], n)
    else:
        lon = rng.uniform(0.0, 360.0, n)
        lat = rng.choice([0.0, 0.5, 12.0, 80.0], n) * rng.uniform(-1, 1, n)
        roll = rng.choice([0.0, 0.0, 20.0, 90.0], n) + rng.uniform(0, 2, n)
    p = synth.pointing_table(lon, lat, 215.0, NPX, NPX, 3.4)
    p[:, 3] = np.deg2rad(roll)
    p[:, 4] *= rng.choice([0.05, 0.4, 0.9, 1.0], n)  # pitch along the rows
    p[:, 6] += rng.uniform(-1.0, 1.0, n)
    p[:, 11] = rng.uniform(0.0, FRAMES - 1.0, n)
    pitch = 215.0 * np.abs(np.tan(p[:, 4])) / (3.0 / N)
    if tied:
        rules = {"min_pitch": float(pitch[0]), "fwd_min_pitch": float(pitch[-1]),
                 "fwd_max_ratio": 0.0}
    else:
        rules = {"min_pitch": float(rng.choice([0.16, 0.5])),
                 "fwd_min_pitch": float(rng.choice([0.3, 0.75, 5.0])),
                 "fwd_max_ratio": float(rng.choice([0.0, 0.02, 0.2]))}
    return p, rules


def _count(layouts, among):
    return len(set(int(v) for v in layouts) & set(among))


@pytest.mark.parametrize("tied", [False, True], ids=["random", "tied"])
@pytest.mark.parametrize("kind", list(KINDS))
def test_passes_match_the_walk_plan(T, kind, tied):
    n_frames, image_kind = KINDS[kind]
    among = (0, 1, 2) if kind == "frames" else (1, 2)
    g = synth.cube_geom(N, 1.5)
    rng = np.random.default_rng(17)
    shape = (N, N, N) if n_frames == 1 else (n_frames, N, N, N)
    ctx, ray = T.Context(), T.Context()
    ray.set_option(T.tomo.TOMO_OPT_PLANE_SYNC, 0)
    kw = {"n_frames": n_frames, "kind": image_kind}
    seen = set()
    for _ in range(60):
        p, rules = _stack(rng, tied)
        x = to_dev(rng.random(shape).astype(np.float32))
        y = to_dev(rng.random((len(p), NPX, NPX)).astype(np.float32))
        T.tomo_set_plane_rules(rules, ctx=ctx)
        ctx.profile(reset=True)
        got = T.tomo_project(x, g, p, NPX, NPX, ctx=ctx, **kw)
        fwd = ctx.profile(reset=True)
        got_t = T.tomo_backproject(y, g, p, ctx=ctx, **kw)
        adj = ctx.profile(reset=True)
        code = T.tomo_walk_plan(len(p), ctx=ctx)
        lat, by_adj, by_fwd = (code >> 5) & 3, (code & 1) != 0, (code & 2) != 0
        copies = _count(lat[by_fwd], among)
        passes = 2 * _count(lat[by_adj], among)
        seen.add((by_fwd.any(), by_fwd.all(), by_adj.any(), copies,
                  2 * copies == passes))
        if tied:
            assert fwd["layout"][0] >= copies
            assert adj["layout"][0] >= passes
        else:
            assert fwd["layout"][0] == copies, (p, rules)
            assert adj["layout"][0] == passes, (p, rules)
            if kind != "B" and by_fwd.any():  # B: one kernel walks both ways
                assert fwd["forward"][0] == (1 if by_fwd.all() else 2)
        assert torch.equal(got, T.tomo_project(x, g, p, NPX, NPX, ctx=ray, **kw))
        want_t = T.tomo_backproject(y, g, p, ctx=ray, **kw)
        torch.testing.assert_close(got_t, want_t, rtol=1e-5,
                                   atol=1e-6 * float(want_t.abs().max()))
    if not tied:
        # every kind of stack was met: none, some and all images by plane, and
        # a forward that copies fewer layouts than the transpose uses
        assert {s[:3] for s in seen} >= {(True, True, True), (True, False, True),
                                         (False, False, True)}
        assert any(s[0] and not s[4] for s in seen)
    ctx.close()
    ray.close()

"""The step of conjugate gradients is not rounded to 32 bits.

The first iterate of CG from 0 is x_1 = alpha b with b = P^T y and
alpha = b.b / b.q, q = P^T P b (normal equations of Eq. criterion, lambda = 0).
b and q come from the public operators, the sums from 64 bits.  Rounding
alpha to float32 moves every voxel of x_1 by the same relative error, up to
2^-24 = 6.0e-8 (at random below that: 9 of 10 data sets are off by more than
3e-9), which CG then amplifies; the float32 rounding of each voxel and the
order of the transpose's additions (~1e-7 per voxel, independent between
110592 voxels) move the ratio by ~3e-10.  The bound is ten times that."""

import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import require_gpu, to_dev

pytestmark = pytest.mark.gpu

N, NPX, N_IMG = 48, 64, 24


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("batched", [False, True], ids=["single", "batched"])
def test_first_step(batched):
    import paper_1103_5904_gb300 as T
    g = synth.cube_geom(N, 1.5)
    ctx = T.Context()
    ratios = []
    for seed in range(8):
        rng = np.random.default_rng(seed)
        p = synth.pointing_table(7.5 * np.arange(N_IMG) + seed, 3.0, 215.0,
                                 NPX, NPX, 3.2)
        y = to_dev((1.0 + rng.random((N_IMG, NPX, NPX))).astype(np.float32))
        if batched:
            x = torch.empty((N, N, N), device="cuda")
            T.tomo_solve_batched([{"geom": g, "pointing": p, "nu": NPX,
                                   "nv": NPX, "images": y, "cube": x,
                                   "lam": 0.0}], 1, ctx=ctx)
        else:
            x, _ = T.tomo_solve(y, g, p, lam=0.0, max_iter=1, ctx=ctx)
        b = T.tomo_backproject(y, g, p, ctx=ctx)
        q = T.tomo_backproject(T.tomo_project(b, g, p, NPX, NPX, ctx=ctx),
                               g, p, ctx=ctx)
        b, q, x = b.double(), q.double(), x.double()
        alpha = (b * b).sum() / (b * q).sum()
        ratios.append(float((x * b).sum() / (b * b).sum() / alpha))
    ctx.close()
    off = np.abs(np.array(ratios) - 1.0)
    assert off.max() < 3e-9, off

"""The work that users of the projector library have it do, as measurable cases.

A case is one call (or, for the differentiable form, one forward and
backward pass) through the public entry points of ``paper_1103_5904_gb300``
on a seeded corona and a seeded set of views.  Sizes are those of the
repository's own workloads (``synth/configs.py``), the ragged ones are
generic.  The keys of a case:

  op        "project" (y = P x), "backproject" (x = P^T y), "gradient" (the
            autograd form, forward and backward), "solve" (CG on one image
            stack) or "solve_batched" (CG on several independent problems)
  nx ny nz  voxels; half: half width of the cube in solar radii
  n_img nu nv  image stack; fov: field of view along u in solar radii
  step      longitude step between views, degrees; second group of views
            `apart` degrees ahead of the first (0: one group)
  lat roll  views take latitudes and rolls in [-lat, lat], [-roll, roll]
  frames    frames of the time-interpolated model (1: static)
  dtype     "f32" or "bf16" cube; kind: "emission", "pB" or "B" images
  occ edge  pixels whose line of sight passes below occ or beyond edge solar
            radii are masked (0: no such limit)
  sphere    radius of the opaque photosphere (0: none)
  shell     voxels below `sphere` and beyond this radius are masked (0: none)
  iters     CG iterations

Views carry what real pointing tables carry: a Carrington longitude that
differs from data set to data set, sub-pixel pointing offsets and one gain
per image.
"""

import math
import random

import numpy as np
import torch

import paper_1103_5904_gb300 as tomo
from paper_1103_5904_gb300 import autograd as tomo_autograd

D_OBS = 215.0   # observer distance (1 AU) in solar radii
LIMB_U = 0.6    # limb darkening of the white-light kinds
LAM = 1e-2      # weight of the smoothness prior in the solvers

_DEFAULTS = {
    "half": 1.5, "fov": 3.2, "step": 1.5, "apart": 0.0, "lat": 0.0,
    "roll": 0.0, "frames": 1, "dtype": "f32", "kind": "emission", "occ": 0.0,
    "edge": 0.0, "sphere": 0.0, "shell": 0.0, "iters": 0,
}


def _case(name, op, n, img, **more):
    c = dict(_DEFAULTS, op=op, nx=n[0], ny=n[1], nz=n[2], n_img=img[0],
             nu=img[1], nv=img[2], **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # A quick look: eight views of a coarse map.  Latency and launches.
        _case("project small", "project", (64, 64, 64), (8, 64, 64),
              step=45.0),
        # A coarse transpose with nothing even about it: rolled, tilted,
        # masked views of a cube of three different sides.
        _case("transpose small ragged", "backproject", (61, 50, 43),
              (7, 75, 53), step=51.0, lat=7.0, roll=15.0, occ=1.0),
        # The repository's CG workload, one projection and one transpose:
        # EUV images of two spacecraft in the ecliptic.
        _case("project ecliptic", "project", (256, 256, 256),
              (240, 512, 512), apart=40.0, occ=1.0),
        _case("transpose ecliptic", "backproject", (256, 256, 256),
              (240, 512, 512), apart=40.0, occ=1.0),
        # Two months of views from near the Earth, whose solar latitude
        # swings by 7 degrees: no view has a cube axis in its rows.
        _case("project tilted", "project", (128, 128, 128), (60, 256, 256),
              step=3.0, lat=7.0, occ=1.0),
        _case("transpose tilted", "backproject", (128, 128, 128),
              (60, 256, 256), step=3.0, lat=7.0, occ=1.0),
        # A gradient step of a learned or smoothed time-dependent map: eight
        # frames, every image between two of them.
        _case("gradient frames", "gradient", (256, 256, 256),
              (120, 512, 512), step=3.0, apart=40.0, frames=8),
        # White-light images of electron density: total brightness with the
        # photosphere and a shell-shaped map, forward and backward.
        _case("gradient white light", "gradient", (256, 256, 256),
              (90, 512, 512), step=4.0, kind="B", occ=1.0, sphere=1.0,
              shell=1.6),
        # The coronagraph workload (512^3), cut to 48 of its 1024^2 images:
        # the forward from a bf16 map, the transpose in float32.
        _case("project coronagraph", "project", (512, 512, 512),
              (48, 1024, 1024), half=4.0, fov=8.0, step=7.0, apart=86.0,
              dtype="bf16", occ=1.5, edge=4.0),
        _case("transpose coronagraph", "backproject", (512, 512, 512),
              (48, 1024, 1024), half=4.0, fov=8.0, step=7.0, apart=86.0,
              occ=1.5, edge=4.0),
        # A map from new observations: ray setup and 20 CG iterations.
        _case("solve", "solve", (128, 128, 128), (60, 256, 256), step=3.0,
              lat=7.0, occ=1.0, iters=20),
        # A set of small inversions (parameter study) in one call.
        dict(_case("solve batched", "solve_batched", (96, 96, 96),
                   (40, 256, 256), iters=10), problems=8, sizes=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["project", "backproject", "project", "backproject",
                     "gradient", "solve", "solve_batched"])
    while True:
        n = _log_int(rng, 40, 512)
        c = _case(None, op, (n, max(8, int(n * rng.uniform(0.7, 1.2))),
                             max(8, int(n * rng.uniform(0.7, 1.2)))),
                  (_log_int(rng, 4, 240), 0, 0))
        c["nu"] = max(16, min(1024, int(n * rng.uniform(0.9, 2.3))))
        c["nv"] = max(16, min(1024, int(c["nu"] * rng.uniform(0.7, 1.3))))
        c["step"] = round(rng.uniform(1.0, 360.0 / c["n_img"]), 3)
        c["apart"] = rng.choice([0.0, 40.0, 86.0])
        c["lat"] = rng.choice([0.0, 0.0, 7.0, 30.0])
        c["roll"] = rng.choice([0.0, 0.0, 10.0])
        c["occ"] = rng.choice([0.0, 1.0])
        if op in ("project", "backproject") and rng.random() < 0.3:
            c["half"], c["fov"], c["occ"], c["edge"] = 4.0, 8.0, 1.5, 4.0
        if op == "project":
            c["dtype"] = rng.choice(["f32", "f32", "bf16"])
        if op == "gradient":
            if rng.random() < 0.5:
                c["frames"] = rng.randint(2, 8)
            else:
                c["kind"] = rng.choice(["pB", "B"])
                c["sphere"], c["shell"] = 1.0, 1.6
        if op == "solve":
            c["iters"] = rng.randint(5, 20)
        if op == "solve_batched":
            c["iters"], c["lat"], c["roll"] = rng.randint(4, 10), 0.0, 0.0
            c["problems"], c["sizes"] = rng.randint(2, 12), rng.randint(2, 99)
            c["nx"] = c["ny"] = c["nz"] = min(n, 128)
            c["nu"] = c["nv"] = min(c["nu"], 256)
            c["n_img"] = min(c["n_img"], 60)
        # no more rays x planes than the largest listed case
        rays = c["n_img"] * c["nu"] * c["nv"] * c.get("problems", 1)
        passes = max(1, 2 * c["iters"])
        if rays * n * passes <= 2.4e10 and n ** 3 * c["frames"] <= 2e8:
            return c


# ------------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _geom(c):
    g = {"r_obs": c["sphere"]}
    for a in "xyz":
        g["n" + a] = c["n" + a]
        g[a + "0"] = -c["half"]
        g["d" + a] = 2.0 * c["half"] / c["n" + a]
    return g


def _pointing(c, rs):
    k = np.arange(c["n_img"])
    lon = c["step"] * k
    if c["apart"]:
        first = (c["n_img"] + 1) // 2
        lon = np.where(k < first, lon, c["apart"] + c["step"] * (k - first))
    cdelt = 2.0 * math.atan(0.5 * c["fov"] / D_OBS) / c["nu"]
    p = np.zeros((c["n_img"], 12))
    p[:, 0] = D_OBS
    p[:, 1] = np.deg2rad(lon + rs.uniform(0.0, 360.0))
    p[:, 2] = np.deg2rad(c["lat"] * rs.uniform(-1.0, 1.0, c["n_img"]))
    p[:, 3] = np.deg2rad(c["roll"] * rs.uniform(-1.0, 1.0, c["n_img"]))
    p[:, 4:6] = cdelt
    p[:, 6] = 0.5 * (c["nu"] - 1) + rs.uniform(-0.5, 0.5, c["n_img"])
    p[:, 7] = 0.5 * (c["nv"] - 1) + rs.uniform(-0.5, 0.5, c["n_img"])
    p[:, 10] = rs.uniform(0.9, 1.1, c["n_img"])
    p[:, 11] = rs.uniform(0.0, c["frames"] - 1.0, c["n_img"])
    return p


def _voxel_centres(c):
    return [torch.linspace(-1.0 + 1.0 / c["n" + a], 1.0 - 1.0 / c["n" + a],
                           c["n" + a], dtype=torch.float64,
                           device=_device()) * c["half"] for a in "xyz"]


def _radius(c):
    x, y, z = _voxel_centres(c)
    return torch.sqrt(z.view(-1, 1, 1) ** 2 + y.view(1, -1, 1) ** 2 +
                      x.view(1, 1, -1) ** 2)


def _corona(c, rs, gen):
    """Density [frames][nz][ny][nx] (one frame: [nz][ny][nx]), float32: a
    radial corona with six streamers and 10 % voxel noise, 0 in the Sun."""
    x, y, z = (v.float() for v in _voxel_centres(c))
    r = _radius(c).float()
    if c["half"] > 2.0:
        bg = r ** -6 + 0.05 * r ** -2
    else:
        bg = torch.exp(-(r - 1.0) / 0.1)
    bg = torch.where(r >= 1.0, bg, torch.zeros_like(bg))
    axes = rs.standard_normal((6, 3))
    axes /= np.linalg.norm(axes, axis=1, keepdims=True)
    phase = rs.uniform(0.0, 2.0 * np.pi, 6)
    out = torch.empty((c["frames"],) + tuple(r.shape), device=r.device)
    out[:] = bg
    for a, ph in zip(axes, phase):
        along = (float(a[0]) * x.view(1, 1, -1) + float(a[1]) *
                 y.view(1, -1, 1) + float(a[2]) * z.view(-1, 1, 1))
        d2 = (r * r - along * along).clamp_(min=0.0)
        beam = torch.where(along > 0.0, bg * torch.exp(d2 * -200.0),
                           torch.zeros_like(bg))
        for f in range(c["frames"]):
            amp = 3.0 * (1.0 + 0.5 * math.sin(2.0 * math.pi * f /
                                              c["frames"] + ph))
            out[f].add_(beam, alpha=amp)
    for f in range(c["frames"]):
        out[f] *= 1.0 + 0.1 * (2.0 * torch.rand(r.shape, generator=gen,
                                                device=r.device) - 1.0)
    return out if c["frames"] > 1 else out[0]


def _tangents(c, p):
    dev = _device()

    def tans(n, cdelt, crpix):
        i = torch.arange(n, dtype=torch.float64, device=dev)
        return torch.tan((i - torch.from_numpy(crpix).to(dev)[:, None]) *
                         torch.from_numpy(cdelt).to(dev)[:, None])
    return tans(c["nu"], p[:, 4], p[:, 6]), tans(c["nv"], p[:, 5], p[:, 7])


def _pixel_mask(c, p):
    if not c["occ"] and not c["edge"]:
        return None
    tu, tv = _tangents(c, p)
    mask = torch.empty((c["n_img"], c["nv"], c["nu"]), dtype=torch.uint8,
                       device=_device())
    for i in range(c["n_img"]):
        t2 = tv[i][:, None] ** 2 + tu[i][None, :] ** 2
        rho = D_OBS * torch.sqrt(t2 / (1.0 + t2))
        out = rho < c["occ"]
        if c["edge"]:
            out |= rho > c["edge"]
        mask[i] = out
    return mask


def _map_mask(c):
    if not c["shell"]:
        return None
    r = _radius(c)
    return ((r < c["sphere"]) | (r > c["shell"])).to(torch.uint8)


def _problem(c, seed):
    """Everything a program has in hand before the call; images for the ops
    that take some."""
    rs = np.random.RandomState(seed % (1 << 32))
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    p = {"geom": _geom(c), "pointing": _pointing(c, rs), "nu": c["nu"],
         "nv": c["nv"]}
    p["mask"] = _pixel_mask(c, p["pointing"])
    p["map_mask"] = _map_mask(c)
    if c["op"] in ("project", "gradient"):
        p["cube"] = _corona(c, rs, gen)
        if c["dtype"] == "bf16":
            p["cube"] = p["cube"].to(torch.bfloat16)
    shape = (c["n_img"], c["nv"], c["nu"])
    if c["op"] in ("backproject", "gradient"):
        # an image of residuals or of an image's cotangent: signed, no pixel
        # alike
        p["images"] = torch.randn(shape, generator=gen, device=_device())
    if c["op"] in ("solve", "solve_batched"):
        # data: the projection of a corona (in 64 bits) with noise, SNR 50
        y = _exact_project(c, p, _corona(c, rs, gen).double())[0]
        y = y.view(shape)
        noise = torch.randn(shape, generator=gen, device=_device())
        y += noise * (y.square().mean().sqrt() / 50.0)
        if p["mask"] is not None:
            y[p["mask"] != 0] = 0.0
        p["images"] = y.float()
    return p


def _subcases(c):
    """The problems of a batch: uneven cube sides, image counts and sizes."""
    rs = np.random.RandomState(c["sizes"])
    out = []
    for _ in range(c["problems"]):
        n = int(c["nx"] * rs.choice([0.33, 0.5, 0.66, 1.0]))
        px = int(c["nu"] * rs.choice([0.25, 0.5, 1.0]))
        n_img = int(c["n_img"] * rs.uniform(0.4, 1.0)) + 1
        out.append(dict(c, nx=n, ny=n, nz=n, nu=px, nv=px, n_img=n_img,
                        step=360.0 / n_img))
    return out


def prepare(case, seed):
    c = dict(_DEFAULTS, **case)
    ctx = tomo.Context()
    if c["op"] != "solve_batched":
        return dict(_problem(c, seed), case=c, ctx=ctx)
    probs = []
    for i, s in enumerate(_subcases(c)):
        p = _problem(s, seed + 1000 * i)
        p["cube"] = torch.empty((s["nz"], s["ny"], s["nx"]), device=_device())
        p["lam"] = LAM
        probs.append(p)
    return {"case": c, "ctx": ctx, "problems": probs}


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["op"] == "solve_batched":
        info = tomo.tomo_solve_batched(state["problems"], c["iters"], ctx=ctx)
        return {"x": [p["cube"] for p in state["problems"]],
                "J": [i["J"].astype(np.float32) for i in info]}
    g, p, nu, nv = state["geom"], state["pointing"], state["nu"], state["nv"]
    if c["op"] == "project":
        return tomo.tomo_project(state["cube"], g, p, nu, nv,
                                 mask=state["mask"], ctx=ctx)
    if c["op"] == "backproject":
        return tomo.tomo_backproject(state["images"], g, p,
                                     mask=state["mask"], ctx=ctx)
    if c["op"] == "gradient":
        x = state["cube"].detach().requires_grad_(True)
        y = tomo_autograd.project(x, g, p, nu, nv, mask=state["mask"],
                                  n_frames=c["frames"], ctx=ctx,
                                  map_mask=state["map_mask"], kind=c["kind"],
                                  limb_u=LIMB_U)
        (grad,) = torch.autograd.grad(y, x, state["images"])
        return {"y": y.detach(), "grad": grad}
    # a new set of observations has new pointings: their rays are set up in
    # the call, as a program that inverts one data set after another has it
    ctx.clear_cache()
    x, info = tomo.tomo_solve(state["images"], g, p, mask=state["mask"],
                              lam=LAM, max_iter=c["iters"], ctx=ctx)
    return {"x": x, "J": info["J"].astype(np.float32)}


# ---------------------------------------------------- work: a lower estimate

def _live_segments(c):
    """(live rays, voxel intersections) of one projection, from a sample of
    rays: every plane of the cube that a line of sight crosses starts a
    voxel."""
    p = _pointing(c, np.random.RandomState(0))
    pick = np.unique(np.linspace(0, c["n_img"] - 1, 12).astype(int))
    iu = np.linspace(0, c["nu"] - 1, min(c["nu"], 48))
    iv = np.linspace(0, c["nv"] - 1, min(c["nv"], 48))
    live = seg = total = 0.0
    for i in pick:
        o, w, e1, e2 = _frame(p[i])
        tu = np.tan((iu - p[i, 6]) * p[i, 4])[None, :, None]
        tv = np.tan((iv - p[i, 7]) * p[i, 5])[:, None, None]
        u = w + tu * e1 + tv * e2
        u /= np.linalg.norm(u, axis=-1, keepdims=True)
        b = u @ o
        rho = np.sqrt(np.maximum(D_OBS ** 2 - b * b, 0.0))
        with np.errstate(divide="ignore"):
            t = np.stack([(s * c["half"] - o) / u for s in (-1, 1)])
        a0 = t.min(0).max(-1)
        a1 = t.max(0).min(-1)
        if c["sphere"]:
            hit = rho < c["sphere"]
            near = -b - np.sqrt(np.maximum(c["sphere"] ** 2 - rho ** 2, 0.0))
            a1 = np.where(hit, np.minimum(a1, near), a1)
        ok = (a1 > a0) & (rho >= c["occ"])
        if c["edge"]:
            ok &= rho <= c["edge"]
        d = 2.0 * c["half"] / np.array([c["nx"], c["ny"], c["nz"]])
        n = np.where(ok, (a1 - a0) * (np.abs(u) / d).sum(-1) + 1.0, 0.0)
        live += ok.sum()
        seg += n.sum()
        total += ok.size
    rays = c["n_img"] * c["nu"] * c["nv"]
    return float(rays * live / total), float(rays * seg / total)


def work(case):
    """Bytes: every input read once and every output written once.  Flops:
    a length (one subtraction) and one multiply-add per intersection, twice
    the multiply-adds where a segment reaches two frames or two sums."""
    c = dict(_DEFAULTS, **case)
    if c["op"] == "solve_batched":
        parts = [work(dict(s, op="solve")) for s in _subcases(c)]
        return {k: sum(q[k] for q in parts) for k in ("bytes", "flops")}
    pixels = c["n_img"] * c["nu"] * c["nv"]
    voxels = c["nx"] * c["ny"] * c["nz"] * c["frames"]
    masks = (pixels if c["occ"] or c["edge"] else 0) + \
        (voxels // c["frames"] if c["shell"] else 0)
    _, seg = _live_segments(c)
    per = 3.0 if c["frames"] == 1 and c["kind"] == "emission" else 5.0
    nbytes = 4.0 * pixels + (2 if c["dtype"] == "bf16" else 4) * voxels + masks
    if c["op"] == "gradient":
        return {"bytes": 2.0 * nbytes, "flops": 2.0 * per * seg}
    if c["op"] == "solve":
        # b, then P and P^T of every iteration; the data and the map once
        return {"bytes": nbytes, "flops": per * seg * (1 + 2 * c["iters"])}
    return {"bytes": nbytes, "flops": per * seg}


# ------------------------------------------- the operators in plain 64 bits

def _frame(q):
    """Observer and image axes of one pointing record: z is the rotation
    axis, the boresight points at Sun centre, e1 = unit(w x z), e2 = e1 x w,
    both turned by the roll."""
    cl, sl, co, so = math.cos(q[2]), math.sin(q[2]), math.cos(q[1]), math.sin(q[1])
    o = q[0] * np.array([cl * co, cl * so, sl])
    w = -o / np.linalg.norm(o)
    a1 = np.cross(w, [0.0, 0.0, 1.0])
    a1 /= np.linalg.norm(a1)
    a2 = np.cross(a1, w)
    cr, sr = math.cos(q[3]), math.sin(q[3])
    return o, w, cr * a1 + sr * a2, -sr * a1 + cr * a2


_TINY = 1e-9  # solar radii: keeps a voxel index inside its cube at the ends


def _rays(c, p, i0, i1):
    """Live rays of images [i0, i1): pixel numbers and the state of a walk."""
    dev = _device()
    ptg = p["pointing"]
    tu, tv = _tangents(c, ptg[i0:i1])
    fr = [_frame(q) for q in ptg[i0:i1]]
    o, w, e1, e2 = (torch.from_numpy(np.stack([f[k] for f in fr])).to(dev)
                    for k in range(4))
    u = (w[:, None, None] + tu[:, None, :, None] * e1[:, None, None] +
         tv[:, :, None, None] * e2[:, None, None])
    u = (u / u.norm(dim=-1, keepdim=True)).view(-1, 3)
    per = c["nu"] * c["nv"]
    img = torch.arange(i0, i1, device=dev).repeat_interleave(per)
    o = o.repeat_interleave(per, 0)
    n = torch.tensor([c["nx"], c["ny"], c["nz"]], device=dev)
    d = 2.0 * c["half"] / n.double()
    t0 = (-c["half"] - o) / u
    t1 = (c["half"] - o) / u
    start = torch.minimum(t0, t1).amax(-1).clamp_(min=0.0)
    end = torch.maximum(t0, t1).amin(-1)
    del t0, t1
    b = (o * u).sum(-1)
    rho2 = (o - b[:, None] * u).square().sum(-1)
    if c["sphere"]:
        near = -b - (c["sphere"] ** 2 - rho2).clamp_(min=0.0).sqrt()
        end = torch.where(rho2 < c["sphere"] ** 2, torch.minimum(end, near), end)
    start, end = start + _TINY, end - _TINY
    live = end > start
    if p["mask"] is not None:
        live &= p["mask"][i0:i1].reshape(-1) == 0
    at = live.nonzero()[:, 0]
    o, u, start, end = o[at], u[at], start[at], end[at]
    cell = torch.floor((o + start[:, None] * u + c["half"]) / d).long()
    cell = torch.minimum(cell.clamp_(min=0), n - 1)
    step = torch.where(u < 0, -1, 1)
    nxt = ((cell + (step > 0)) * d - c["half"] - o) / u
    stride = torch.tensor([1, c["nx"], c["nx"] * c["ny"]], device=dev)
    return {"pix": at + i0 * per, "img": img[at], "rho2": rho2[at],
            "t": start, "end": end, "idx": (cell * stride).sum(-1),
            "next": [nxt[:, k].contiguous() for k in range(3)],
            "dt": [(d[k] / u[:, k].abs()) for k in range(3)],
            "jump": [(step[:, k] * stride[k]) for k in range(3)]}


def _walk(r):
    """Siddon's intersections of the rays, one voxel of every ray at a time:
    yields (voxel, length); finished rays yield length 0."""
    t, end, idx, nxt = r["t"], r["end"], r["idx"], r["next"]
    k = 0
    while t.numel() and (k % 16 or bool((t < end).any())):
        first = torch.minimum(torch.minimum(nxt[0], nxt[1]), nxt[2])
        to = torch.minimum(first, end)
        yield idx, to - t
        t = to
        todo = first < end
        for a in range(3):
            here = (nxt[a] == first) & todo
            todo = todo & ~here
            nxt[a] = torch.where(here, nxt[a] + r["dt"][a], nxt[a])
            idx = torch.where(here, idx + r["jump"][a], idx)
        k += 1


def _chunks(c, p):
    per = max(1, 2_000_000 // (c["nu"] * c["nv"]))
    for i0 in range(0, c["n_img"], per):
        r = _rays(c, p, i0, min(c["n_img"], i0 + per))
        gain = torch.from_numpy(p["pointing"][:, 10]).to(_device())
        r["gain"] = gain[r["img"]]
        if c["frames"] > 1:
            tau = torch.from_numpy(p["pointing"][:, 11]).to(_device())[r["img"]]
            r["frame"] = tau.floor().long().clamp_(0, c["frames"] - 2)
            r["w"] = tau - r["frame"]
        yield r


def _exact_project(c, p, *cubes):
    """P x in 64 bits for every cube given, one flat image stack each."""
    n = c["nx"] * c["ny"] * c["nz"]
    flat = [x.reshape(-1) for x in cubes]
    out = [torch.zeros(c["n_img"] * c["nu"] * c["nv"], dtype=torch.float64,
                       device=_device()) for _ in cubes]
    for r in _chunks(c, p):
        acc = [torch.zeros_like(r["t"]) for _ in cubes]
        for idx, length in _walk(r):
            for a, x in zip(acc, flat):
                if c["frames"] > 1:
                    i = idx + n * r["frame"]
                    v = torch.lerp(x[i], x[i + n], r["w"])
                else:
                    v = x[idx]
                a.addcmul_(length, v)
        for y, a in zip(out, acc):
            y[r["pix"]] = r["gain"] * a
    return out


def _exact_backproject(c, p, *images):
    """P^T y in 64 bits for every image stack given, one flat map each."""
    n = c["nx"] * c["ny"] * c["nz"]
    flat = [y.reshape(-1) for y in images]
    out = [torch.zeros(n * c["frames"], dtype=torch.float64, device=_device())
           for _ in images]
    for r in _chunks(c, p):
        gy = [r["gain"] * y[r["pix"]] for y in flat]
        for idx, length in _walk(r):
            for x, g in zip(out, gy):
                if c["frames"] > 1:
                    i = idx + n * r["frame"]
                    x.index_add_(0, i, length * g * (1.0 - r["w"]))
                    x.index_add_(0, i + n, length * g * r["w"])
                else:
                    x.index_add_(0, idx, length * g)
    return out


def _thomson(c):
    """(m, m') at the voxel centres: van de Hulst's coefficients with
    sin(Omega) = 1 / r and the limb darkening, 0 inside the Sun."""
    r = _radius(c)
    far = r > 1.0
    r = torch.where(far, r, torch.full_like(r, 2.0))
    s = 1.0 / r
    q = torch.sqrt(1.0 - s * s)
    g = q * q / s * torch.log((1.0 + s) / q)
    c1 = q * s * s
    c2 = -(1.0 - 3.0 * s * s - g * (1.0 + 3.0 * s * s)) / 8.0
    c3 = 4.0 / 3.0 - q - q ** 3 / 3.0
    c4 = (5.0 + s * s - g * (5.0 - s * s)) / 8.0
    m = ((1.0 - LIMB_U) * c1 + LIMB_U * c2) / r ** 4
    m2 = 2.0 * ((1.0 - LIMB_U) * c3 + LIMB_U * c4) / r ** 2
    zero = torch.zeros_like(r)
    return torch.where(far, m, zero), torch.where(far, m2, zero)


def _impact2(c, p):
    out = torch.zeros(c["n_img"] * c["nu"] * c["nv"], dtype=torch.float64,
                      device=_device())
    for r in _chunks(c, p):
        out[r["pix"]] = r["rho2"]
    return out


def _exact_gradient(c, p):
    shape = (c["n_img"], c["nv"], c["nu"])
    x, y = p["cube"].double(), p["images"].double()
    keep = 1.0 if p["map_mask"] is None else (p["map_mask"] == 0).double()
    if c["kind"] == "emission":
        out = _exact_project(c, p, x * keep)[0]
        grad = _exact_backproject(c, p, y)[0].view(x.shape) * keep
    else:
        m, m2 = _thomson(c)
        rho2 = _impact2(c, p)
        a, b = _exact_project(c, p, x * keep * m, x * keep * m2)
        out = rho2 * a if c["kind"] == "pB" else b - rho2 * a
        ga, gb = _exact_backproject(c, p, rho2 * y.reshape(-1), y)
        grad = m * ga.view(x.shape)
        if c["kind"] == "B":
            grad = m2 * gb.view(x.shape) - grad
        grad = grad * keep
    return {"y": out.view(shape), "grad": grad}


def _prior(x):
    """D^T D x, D the forward differences along the three axes."""
    q = torch.zeros_like(x)
    for a in range(3):
        n = x.shape[a]
        if n > 1:
            d = x.narrow(a, 1, n - 1) - x.narrow(a, 0, n - 1)
            q.narrow(a, 1, n - 1).add_(d)
            q.narrow(a, 0, n - 1).sub_(d)
    return q


def _exact_solve(c, p):
    """Conjugate gradients on (P^T P + LAM D^T D) x = P^T y from 0, and the
    criterion of every iterate."""
    shape = (c["nz"], c["ny"], c["nx"])
    y = p["images"].double()
    yy = y.square().sum() if p["mask"] is None else \
        y[p["mask"] == 0].square().sum()
    b = _exact_backproject(c, p, y)[0].view(shape)
    x, r = torch.zeros_like(b), b.clone()
    d, rr = r.clone(), r.square().sum()
    crit = [yy]
    for _ in range(c["iters"]):
        q = _exact_backproject(c, p, _exact_project(c, p, d)[0])[0].view(shape)
        q += LAM * _prior(d)
        alpha = rr / (d * q).sum()
        x += alpha * d
        r -= alpha * q
        new = r.square().sum()
        d = r + (new / rr) * d
        rr = new
        crit.append(yy - (x * (r + b)).sum())
    return x, torch.stack(crit)


def exact(case, seed):
    c = dict(_DEFAULTS, **case)
    if c["op"] == "solve_batched":
        got = [_exact_solve(s, _problem(s, seed + 1000 * i))
               for i, s in enumerate(_subcases(c))]
        return {"x": [g[0] for g in got], "J": [g[1] for g in got]}
    p = _problem(c, seed)
    if c["op"] == "project":
        return _exact_project(c, p, p["cube"].double())[0].view(
            c["n_img"], c["nv"], c["nu"])
    if c["op"] == "backproject":
        return _exact_backproject(c, p, p["images"].double())[0].view(
            c["nz"], c["ny"], c["nx"])
    if c["op"] == "gradient":
        return _exact_gradient(c, p)
    x, crit = _exact_solve(c, p)
    return {"x": x, "J": crit}


if __name__ == "__main__":
    for one in listed() + [draw(random.Random(s)) for s in range(6)]:
        print(one, work(one))

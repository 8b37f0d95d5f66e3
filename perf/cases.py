"""The work this library is run for, as cases that can be timed and checked.

The inputs follow the paper-shaped flights of the repository's benchmark and
tests: an 8176 x 6132 px camera of 15625 px focal length 300 m over terrain
with buildings, strips of 80 % forward and 60 % side overlap, Brown distortion
per image, 0.5 px noise with 2 % outliers of +-50 px, GNSS priors of 5 cm, IMU
priors of 0.01 degrees, points known to 10 cm.

A solve hands back the whole state it adjusted: rotations, centres, points.
BA_FP64 works in binary64 and its state is taken as such.  BA_MIXED computes
its steps in binary32 from whitened residuals of that type, so the program
takes its state as binary32 values: the digits beyond them follow the order
of the sums, which the interface leaves to the launch parameters.
"""
import ctypes
import math
import random
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2511_06152_gb300 as ba

WIDTH, HEIGHT, FOCAL, ALTITUDE = 8176, 6132, 15625.0, 300.0
ACROSS, ALONG = WIDTH * ALTITUDE / FOCAL, HEIGHT * ALTITUDE / FOCAL  # footprint, metres
BASE, SPACING = 0.2 * ALONG, 0.4 * ACROSS                           # between exposures, between strips
SIGMA_PX, HUBER_PX, SIGMA_GNSS, SIGMA_IMU = 0.5, 1.0, 0.05, math.radians(0.01)
MU0 = 1e-4


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one local cluster of 2 strips x 3 images at the smallest configured size, in binary64, 10 iterations:
        # launches and latency only
        dict(name="run_small_fp64", kind="run", precision="fp64", strips=2, images=6, points=2000, track="all",
             fixed=0, iters=10),
        # one LM step of a sliding window whose first images are held fixed: the caller who looks at every step
        dict(name="step_window_mixed", kind="run", precision="mixed", strips=3, images=16, points=15000, track="all",
             fixed=2, iters=1),
        # the paper-scale cluster, 24 images and about 230 k observations, solved on its own
        dict(name="run_cluster_mixed", kind="run", precision="mixed", strips=3, images=24, points=40000, track="all",
             fixed=0, iters=20),
        # the same in binary64, for callers who want the parity path
        dict(name="run_cluster_fp64", kind="run", precision="fp64", strips=3, images=24, points=40000, track="all",
             fixed=0, iters=5),
        # a few uneven clusters at once: what one flight's windows give
        dict(name="batch_12_mixed", kind="batch", precision="mixed", clusters=12, iters=20),
        # many uneven clusters of 8-32 images and 5k-60k points at once: the offline workload, and the largest
        dict(name="batch_128_mixed", kind="batch", precision="mixed", clusters=128, iters=20),
        # a whole flight of 3 x 40 images as one cluster (n = 720): the global reference solution
        dict(name="flight_120_mixed", kind="run", precision="mixed", strips=3, images=120, points=100001, track="all",
             fixed=0, iters=3),
        # a block of 10 x 40 images (n = 2400) with sparse tracks
        dict(name="block_400_mixed", kind="run", precision="mixed", strips=10, images=400, points=200000,
             track="long", fixed=0, iters=3),
        # a window's whole life from host arrays: created, solved, read back with its reprojection errors, freed
        dict(name="window_whole_mixed", kind="window", precision="mixed", strips=3, images=20, points=33001,
             track="all", fixed=3, iters=10),
        # windows of several flights through the serving scheduler
        dict(name="serve_16_mixed", kind="serve", precision="mixed", clusters=16, iters=10),
        # the robust cost of a caller's device arrays, for callers that cannot allocate
        dict(name="cost_120_images", kind="cost", strips=3, images=120, points=150000),
        # cluster formation and tracking: footprints on the surface model, their overlaps, and image 0's patch
        # grid moved to 40 images
        dict(name="formation_120", kind="formation", strips=3, images=120, cell=2.0, grid_x=128, grid_y=96,
             targets=40),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Weights by use: solves first, then serving, whole windows, and the calls around them."""
    kind = rng.choice(["run", "run", "run", "batch", "batch", "large", "window", "serve", "cost", "formation"])
    if kind == "run":
        strips = rng.choice([1, 2, 3])
        images = rng.randint(max(3, 2 * strips), 32)
        track = rng.choice(["all", "geometric"])
        fixed = rng.choice([0, 0, 1, min(4, images // 3)])
        if rng.random() < 0.3:
            return dict(kind="run", precision="fp64", strips=strips, images=images, points=_log(rng, 300, 40000),
                        track=track, fixed=fixed, iters=rng.choice([1, 3, 5]))
        return dict(kind="run", precision="mixed", strips=strips, images=images, points=_log(rng, 300, 60000),
                    track=track, fixed=fixed, iters=rng.choice([1, 10, 20]))
    if kind == "batch":
        return dict(kind="batch", precision="mixed", clusters=_log(rng, 2, 120), iters=rng.choice([10, 20]))
    if kind == "large":
        images = _log(rng, 34, 380)
        strips = rng.choice([2, 3, 4]) if images < 160 else rng.choice([6, 8, 10])
        return dict(kind="run", precision="mixed", strips=strips, images=images, points=images * rng.randint(200, 500),
                    track=rng.choice(["all", "long"]) if images < 130 else "long", fixed=rng.choice([0, 3]),
                    iters=rng.choice([1, 3]))
    if kind == "window":
        return dict(kind="window", precision="mixed", strips=rng.choice([2, 3]), images=rng.randint(12, 32),
                    points=_log(rng, 5000, 50000), track="all", fixed=rng.choice([0, 2, 4]), iters=10)
    if kind == "serve":
        return dict(kind="serve", precision="mixed", clusters=rng.randint(2, 48), iters=10)
    if kind == "cost":
        images = _log(rng, 6, 400)
        return dict(kind="cost", strips=rng.choice([1, 2, 3]) if images < 130 else 10, images=images,
                    points=images * rng.randint(100, 1200))
    return dict(kind="formation", strips=rng.choice([2, 3, 4]), images=rng.randint(8, 200), cell=rng.choice([1.0, 2.0, 5.0]),
                grid_x=rng.randint(16, 128), grid_y=rng.randint(12, 96), targets=rng.randint(1, 40))


# ------------------------------------------------------------------ scenes, made on the GPU

def _gen(*seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.SeedSequence([int(s) & 0x7fffffff for s in seed]).generate_state(1)[0]))
    return g


def _uniform(g, lo, hi, n):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _hat(w):
    z = torch.zeros_like(w[..., 0])
    x, y, s = w.unbind(-1)
    return torch.stack([z, -s, y, s, z, -x, -y, x, z], -1).reshape(*w.shape[:-1], 3, 3)


def _exp(w):
    """Rotation matrices of rotation vectors (Rodrigues)."""
    t2 = (w * w).sum(-1)[..., None, None]
    t = t2.sqrt()
    small = t2 < 1e-16
    one = torch.ones_like(t)
    a = torch.where(small, 1 - t2 / 6, torch.sin(t) / torch.where(small, one, t))
    b = torch.where(small, 0.5 - t2 / 24, (1 - torch.cos(t)) / torch.where(small, one, t2))
    K = _hat(w)
    return torch.eye(3, dtype=w.dtype, device=w.device) + a * K + b * (K @ K)


def _boxes(g, x0, x1, y0, y1):
    """Flat-roofed buildings, about one in 2500 square metres."""
    n = max(1, int((x1 - x0) * (y1 - y0) / 2500.0))
    cx, cy = _uniform(g, x0, x1, n), _uniform(g, y0, y1, n)
    hw, hh = _uniform(g, 5.0, 20.0, n), _uniform(g, 5.0, 20.0, n)
    return torch.stack([cx - hw, cx + hw, cy - hh, cy + hh, _uniform(g, 5.0, 30.0, n)], 1)


def _ground(x, y, boxes):
    w = 2 * math.pi
    z = 20.0 * (torch.sin(w * x / 400.0) + torch.sin(w * y / 250.0) + torch.sin(w * (x + y) / 600.0)) / 3.0
    for i in range(0, x.numel(), 1 << 17):
        a, b = x[i:i + (1 << 17), None], y[i:i + (1 << 17), None]
        hit = (a >= boxes[:, 0]) & (a <= boxes[:, 1]) & (b >= boxes[:, 2]) & (b <= boxes[:, 3])
        z[i:i + (1 << 17)] += torch.where(hit, boxes[:, 4], 0.0).max(1).values
    return z


def _flight(g, strips, images):
    """Cameras of serpentine strips: intrinsics, true rotations and centres, buildings, the ground's extent."""
    per = -(-images // strips)
    place = []
    for s in range(strips):
        order = range(per) if s % 2 == 0 else range(per - 1, -1, -1)
        place += [((s - (strips - 1) / 2) * SPACING, (i - (per - 1) / 2) * BASE, 1.0 if s % 2 == 0 else -1.0)
                  for i in order]
    place = torch.tensor(place[:images], dtype=torch.float64, device="cuda")
    n, c = images, place[:, 2]
    zero = torch.zeros_like(c)
    nadir = torch.stack([c, zero, zero, zero, -c, zero, zero, zero, -torch.ones_like(c)], 1).reshape(n, 3, 3)
    R = nadir @ _exp(math.radians(0.5) * _normal(g, n, 3))
    T = torch.cat([place[:, :2], torch.full((n, 1), ALTITUDE, dtype=torch.float64, device="cuda")], 1)
    T = T + _normal(g, n, 3) * torch.tensor([0.5, 0.5, 1.0], dtype=torch.float64, device="cuda")
    intr = torch.zeros(n, 7, dtype=torch.float64, device="cuda")
    intr[:, 0], intr[:, 1], intr[:, 2] = FOCAL, WIDTH / 2.0, HEIGHT / 2.0
    intr[:, 3:] = 1e-3 * _normal(g, n, 4)
    pad = ACROSS / 2 + 10.0
    ext = [float(T[:, 0].min()) - pad, float(T[:, 0].max()) + pad, float(T[:, 1].min()) - pad,
           float(T[:, 1].max()) + pad]
    return intr, R, T, _boxes(g, *ext), ext


def _project(intr, Xc):
    """Pixels of camera-frame points (intr [..., 7], Xc [..., 3])."""
    a, b = Xc[..., 0] / Xc[..., 2], Xc[..., 1] / Xc[..., 2]
    f, cx, cy, k1, k2, p1, p2 = intr.unbind(-1)
    r2 = a * a + b * b
    rad = 1 + r2 * (k1 + k2 * r2)
    u = f * (a * rad + 2 * p1 * a * b + p2 * (r2 + 2 * a * a)) + cx
    v = f * (b * rad + p1 * (r2 + 2 * b * b) + 2 * p2 * a * b) + cy
    return u, v


def _observe(g, intr, R, T, X, track):
    """For points X: the images that observe each (bool [n, images]); points of fewer than two views observe none."""
    Xc = torch.einsum("nci,cij->ncj", X[:, None, :] - T, R)
    u, v = _project(intr, Xc)
    vis = (Xc[..., 2] > 1.0) & (u >= 0) & (u < WIDTH) & (v >= 0) & (v < HEIGHT)
    seen = vis.sum(1)
    if track != "all":  # track length 2 + geometric, truncated; the images drawn among those that see the point
        p, most = (0.5, 8) if track == "geometric" else (0.25, 16)
        more = torch.rand(len(X), generator=g, device="cuda", dtype=torch.float64)
        length = 2 + torch.floor(torch.log1p(-more) / math.log(1 - p)).long()
        length = torch.minimum(length.clamp(max=most), seen)
        key = torch.rand(vis.shape, generator=g, device="cuda") + 2.0 * (~vis)
        k = min(most, vis.shape[1])
        first = torch.topk(key, k, dim=1, largest=False, sorted=True).indices
        take = torch.arange(k, device="cuda") < length[:, None]
        vis = torch.zeros_like(vis).scatter_(1, first, take)
    return vis & (seen >= 2)[:, None]


def _scene(seed, strips, images, points, track, fixed=0, device_arrays=False, obs=None):
    """One cluster as the arrays a caller has: host arrays, or device tensors.  obs: that many observations, the
    rest missed by the tracker (third and later views of a point first)."""
    g = _gen(*np.atleast_1d(seed))
    intr, R, T, boxes, ext = _flight(g, strips, images)
    step = max(1024, min(points + points // 2 + 512, (1 << 23) // images))
    X, cam, pt, have = [], [], [], 0
    while have < points:
        x, y = _uniform(g, ext[0], ext[1], step), _uniform(g, ext[2], ext[3], step)
        Y = torch.stack([x, y, _ground(x, y, boxes)], 1)
        vis = _observe(g, intr, R, T, Y, track)
        keep = torch.nonzero(vis.any(1))[:points - have, 0]
        p, c = torch.nonzero(vis[keep], as_tuple=True)  # sorted by point, then image
        X.append(Y[keep])
        cam.append(c)
        pt.append(p + have)
        have += len(keep)
    X, cam, pt = torch.cat(X), torch.cat(cam), torch.cat(pt)
    if obs is not None:
        first = torch.searchsorted(pt, pt)  # each observation's point starts there
        view = torch.arange(len(pt), device="cuda") - first
        key = torch.rand(len(pt), generator=g, device="cuda", dtype=torch.float64) - (view < 2).double()
        if len(pt) < obs:
            raise ValueError("fewer observations than wanted")
        keep = torch.sort(torch.argsort(key)[:obs]).values
        cam, pt = cam[keep], pt[keep]
    u, v = _project(intr[cam], torch.einsum("ni,nij->nj", X[pt] - T[cam], R[cam]))
    n = len(cam)
    noise = SIGMA_PX * _normal(g, n, 2)
    out = torch.rand(n, generator=g, device="cuda") < 0.02
    noise = torch.where(out[:, None], 100.0 * torch.rand(n, 2, generator=g, device="cuda", dtype=torch.float64) - 50.0,
                        noise)
    Tp = T + SIGMA_GNSS * _normal(g, images, 3)
    Rp = R @ _exp(SIGMA_IMU * _normal(g, images, 3))
    hold = torch.zeros(images, dtype=torch.uint8, device="cuda")
    hold[:fixed] = 1
    held = hold.bool()
    sc = dict(intr=intr, R0=torch.where(held[:, None, None], R, Rp).reshape(images, 9),
              T0=torch.where(held[:, None], T, Tp), X0=X + 0.1 * _normal(g, points, 3), R_prior=Rp.reshape(images, 9),
              T_prior=Tp, fixed=hold, obs_cam=cam.to(torch.int32), obs_pt=pt.to(torch.int32),
              obs_uv=torch.stack([u, v], 1) + noise)
    if not device_arrays:
        sc = {k: t.cpu().numpy() for k, t in sc.items()}
    sc.update(n_cams=images, n_pts=points, n_obs=n, sigma_px=SIGMA_PX, huber_delta=HUBER_PX, sigma_gnss=SIGMA_GNSS,
              sigma_imu=SIGMA_IMU, mu0=MU0)
    return sc


def _specs(case, seed):
    """The uneven clusters of a batch: 8-32 images in 2-3 strips, 5k-60k points of short tracks; windows through
    the scheduler: 12-32 images, dense tracks, the first ones held fixed.  Their sizes are the case's own, whatever
    the seed."""
    r = random.Random(1009 + case["clusters"])
    out = []
    for i in range(case["clusters"]):
        if case["kind"] == "batch":
            out.append(dict(seed=(seed, i), strips=r.choice([2, 3]), images=r.randint(8, 32),
                            points=r.randint(5000, 60000), track="geometric"))
        else:
            n = r.randint(12, 32)
            out.append(dict(seed=(seed, i), strips=3, images=n, points=n * 1000 + r.randint(0, 999), track="all",
                            fixed=r.randint(0, n // 8)))
    return out


def _scenes(case, seed):
    if case["kind"] in ("batch", "serve"):
        return [_scene(**s) for s in _specs(case, seed)]
    obs = int(0.85 * _views(case)[0] * case["points"]) if case["kind"] == "window" else None
    return [_scene(seed, case["strips"], case["images"], case["points"], case["track"], case["fixed"], obs=obs)]


# ------------------------------------------------------------------ states and passes

class _State:
    """What the program holds between passes; its context goes with it."""

    def __init__(self, case):
        self.case = case
        self.mixed = case.get("precision") == "mixed"
        self.ctx = None

    def open(self, **kw):
        # the context works on a stream of the program's own
        self.stream = torch.cuda.Stream()
        self.ctx = ba.Context(precision=ba.BA_MIXED if self.mixed else ba.BA_FP64, stream=self.stream.cuda_stream, **kw)

    def __del__(self):
        if self.ctx is not None:
            self.ctx.close()


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "cost":
        s.scene = _scene(seed, case["strips"], case["images"], case["points"], "all", 2, device_arrays=True)
        s.F = torch.zeros(1, dtype=torch.float64, device="cuda")
        d = ba.ba_cluster_desc()
        d.n_cams, d.n_pts, d.n_obs, d.ptr_kind = case["images"], case["points"], s.scene["n_obs"], ba.BA_PTR_DEVICE
        for field, key, of in (("intr", "intr", ctypes.c_double), ("R", "R0", ctypes.c_double),
                               ("T", "T0", ctypes.c_double), ("X", "X0", ctypes.c_double),
                               ("R_prior", "R_prior", ctypes.c_double), ("T_prior", "T_prior", ctypes.c_double),
                               ("fixed", "fixed", ctypes.c_uint8), ("obs_cam", "obs_cam", ctypes.c_int32),
                               ("obs_pt", "obs_pt", ctypes.c_int32), ("obs_uv", "obs_uv", ctypes.c_double)):
            s.scene[key] = s.scene[key].contiguous()
            setattr(d, field, ctypes.cast(s.scene[key].data_ptr(), ctypes.POINTER(of)))
        d.sigma_px, d.huber_delta_px, d.sigma_gnss_m, d.sigma_imu_rad = SIGMA_PX, HUBER_PX, SIGMA_GNSS, SIGMA_IMU
        s.desc = d
        return s
    if kind == "formation":
        s.inputs = _formation_inputs(case, seed)
        s.open()
        return s
    if kind == "window":
        s.scene = _scenes(case, seed)[0]
        s.open()
        return s
    scenes = _scenes(case, seed)
    s.open(**({"n_slots": 64} if kind == "serve" else {}))
    with ThreadPoolExecutor(8) as pool:  # creation takes host time only: a program creates on several threads
        s.ids = list(pool.map(s.ctx.create_cluster, scenes))
    if kind == "run":
        return s
    # many clusters: the program keeps their states on the GPU, one array for all rotations, centres and points
    s.sizes = [(x["n_cams"], x["n_pts"]) for x in scenes]
    nc, npt = sum(a for a, _ in s.sizes), sum(b for _, b in s.sizes)
    s.R, s.T, s.X = (torch.zeros(n, w, dtype=torch.float64, device="cuda") for n, w in ((nc, 9), (nc, 3), (npt, 3)))
    torch.cuda.synchronize()
    return s


def _read_states(s):
    """Every cluster's state into the program's device arrays (the C entry point with device pointers)."""
    at = lambda t, row: ctypes.cast(t.data_ptr() + 8 * t.shape[1] * row, ctypes.POINTER(ctypes.c_double))  # noqa: E731
    c = p = 0
    for cid, (nc, npt) in zip(s.ids, s.sizes):
        if s.ctx.L.ba_get_state(s.ctx.h, cid, at(s.R, c), at(s.T, c), at(s.X, p), ba.BA_PTR_DEVICE) != ba.BA_OK:
            raise RuntimeError("ba_get_state")
        c += nc
        p += npt
    with torch.cuda.stream(s.stream):
        return [t.float() if s.mixed else t for t in (s.R, s.T, s.X)]


def run(s):
    case, ctx, kind = s.case, s.ctx, s.case["kind"]
    if kind == "run":
        cid = s.ids[0]
        ctx.reset_batch(s.ids)  # every pass solves from the initial state
        if case["iters"] == 1:
            ctx.solve_step(cid)
        else:
            ctx.run(cid, case["iters"], trace=False)
        return [a.astype(np.float32) if s.mixed else a for a in ctx.get_state(cid)]
    if kind == "batch":
        ctx.reset_batch(s.ids)
        res = ctx.solve_batch(s.ids, case["iters"])
        cost = np.array([r["final_cost"] for r in res])
        return _read_states(s) + [cost.astype(np.float32) if s.mixed else cost]
    if kind == "serve":
        ctx.reset_batch(s.ids)
        wait = [ctx.submit(c, case["iters"]) for c in s.ids]
        cost = np.zeros(len(wait))
        for i, t in enumerate(wait):
            while (r := ctx.poll(t)) is None:
                time.sleep(5e-5)
            cost[i] = r["final_cost"]
        return _read_states(s) + [cost.astype(np.float32)]
    if kind == "window":
        cid = ctx.create_cluster(s.scene)
        ctx.run(cid, case["iters"], trace=False)
        got = ctx.get_state(cid)
        err = ctx.reprojection_errors(cid)
        ctx.destroy_cluster(cid)
        return [a.astype(np.float32) for a in got] + [err.astype(np.float32)]
    if kind == "cost":
        if ba.lib().ba_cost_noalloc(ctypes.byref(s.desc), torch.cuda.current_stream().cuda_stream,
                                    ctypes.cast(s.F.data_ptr(), ctypes.POINTER(ctypes.c_double))) != ba.BA_OK:
            raise RuntimeError("ba_cost_noalloc")
        return s.F
    f = s.inputs
    corners = ctx.footprints(f["intr"], WIDTH, HEIGHT, f["R"], f["T"], f["dsm"])
    area = ctx.footprint_overlaps(corners, corners)
    m = slice(1, 1 + case["targets"])
    p, inside = ctx.patch_transfer_poses(f["p0"], f["intr"][0], f["R"][0], f["T"][0], f["depth"], f["intr"][m],
                                         f["R"][m], f["T"][m], WIDTH, HEIGHT)
    return [corners, area, p, inside]


def _formation_inputs(case, seed):
    g = _gen(seed, case["images"], 77)
    n = max(case["images"], case["targets"] + 1)
    intr, R, T, boxes, ext = _flight(g, case["strips"], n)
    cell = case["cell"]
    nx, ny = int((ext[1] - ext[0]) / cell) + 2, int((ext[3] - ext[2]) / cell) + 2
    xs = ext[0] + cell * torch.arange(nx, dtype=torch.float64, device="cuda")
    ys = ext[2] + cell * torch.arange(ny, dtype=torch.float64, device="cuda")
    y, x = torch.meshgrid(ys, xs, indexing="ij")
    h = _ground(x.reshape(-1).clone(), y.reshape(-1).clone(), boxes).reshape(ny, nx).cpu().numpy()
    px = (np.arange(case["grid_x"]) + 0.5) * WIDTH / case["grid_x"]
    py = (np.arange(case["grid_y"]) + 0.5) * HEIGHT / case["grid_y"]
    p0 = np.stack(np.meshgrid(px, py), -1).reshape(-1, 2)
    return dict(intr=intr.cpu().numpy(), R=R.reshape(n, 9).cpu().numpy(), T=T.cpu().numpy(), p0=p0,
                depth=float(T[0, 2].cpu()) - float(h.mean()),
                dsm=dict(h=h, x0=ext[0], y0=ext[2], dx=cell, dy=cell))


# ------------------------------------------------------------------ work

def _views(case):
    """Observations and co-visible observation pairs of a point, on average."""
    if case["kind"] == "batch" or case.get("track") == "geometric":
        return 2.62, 2.6
    if case.get("track") == "long":
        return 4.6, 10.0
    strips, images = case.get("strips", 3), case.get("images", 22)
    per = -(-images // strips)
    v = max(2.0, images * ACROSS * ALONG / (((strips - 1) * SPACING + ACROSS) * ((per - 1) * BASE + ALONG)))
    return v, 0.6 * v * (v - 1)


def work(case):
    kind = case["kind"]
    if kind == "formation":
        n, q, m = case["images"], case["grid_x"] * case["grid_y"], case["targets"]
        nodes = (n / case["strips"] * BASE + ACROSS) * (case["strips"] * SPACING + ACROSS) / case["cell"] ** 2
        return {"bytes": 8.0 * (nodes + 19 * n + 12 * n + n * n) + q * 16.0 + q * m * 17.0,
                "flops": 45.0 * q * m + 300.0 * n * n + 4.0 * n * 90 * 40}
    if kind in ("batch", "serve"):
        k, points, images = case["clusters"], 32500.0, 20.0
        if kind == "serve":
            points, images = 22500.0, 22.0
    else:
        k, points, images = 1, case["points"], case["images"]
    v, pairs = _views(case)
    obs = points * v
    if kind == "cost":
        return {"bytes": 24.0 * obs + 24.0 * points + 152.0 * images, "flops": 70.0 * obs}
    n = 6.0 * images
    band = n if images <= 32 else min(n, 6.0 * 12 * case["strips"])
    flops = case["iters"] * (obs * (258 + 294 + 236 + 36) + 216 * pairs * points + 75 * points + n * band * band / 3)
    return {"bytes": k * (24.0 * obs + 48.0 * points + 400.0 * images + (8.0 * obs if kind == "window" else 0.0)),
            "flops": k * flops}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch

def _log3(E):
    v = 0.5 * torch.stack([E[:, 2, 1] - E[:, 1, 2], E[:, 0, 2] - E[:, 2, 0], E[:, 1, 0] - E[:, 0, 1]], 1)
    s = v.norm(dim=1)
    t = torch.atan2(s, 0.5 * (E.diagonal(dim1=1, dim2=2).sum(1) - 1))
    return v * torch.where(s > 1e-12, t / s.clamp(min=1e-300), torch.ones_like(s))[:, None]


class _Problem:
    """Levenberg-Marquardt on one cluster as the interface states it: Huber on the squared residual norm, GNSS and
    IMU priors of the free images, Marquardt scaling, Nielsen's damping; points eliminated, dense solve."""

    def __init__(self, sc):
        dev = lambda k: torch.as_tensor(sc[k], device="cuda")  # noqa: E731
        self.intr, self.Rp, self.Tp = dev("intr"), dev("R_prior").reshape(-1, 3, 3), dev("T_prior")
        self.cam, self.pt, self.uv = dev("obs_cam").long(), dev("obs_pt").long(), dev("obs_uv")
        self.R, self.T, self.X = dev("R0").reshape(-1, 3, 3).clone(), dev("T0").clone(), dev("X0").clone()
        self.free = torch.nonzero(dev("fixed") == 0)[:, 0]
        self.nf, self.np = len(self.free), len(self.X)
        self.fi = torch.full((len(self.R),), -1, device="cuda")
        self.fi[self.free] = torch.arange(self.nf, device="cuda")
        # pairs of observations of one point, both images free (observations are sorted by point)
        a, b, d, f = [], [], 1, self.fi[self.cam] >= 0
        while True:
            same = self.pt[d:] == self.pt[:-d]
            if d >= len(self.pt) or not bool(same.any()):
                break
            i = torch.nonzero(same & f[d:] & f[:-d])[:, 0]
            a.append(i)
            b.append(i + d)
            d += 1
        self.pair = (torch.cat(a), torch.cat(b)) if a else None

    def residual(self, R, T, X):
        Xc = torch.einsum("ni,nij->nj", X[self.pt] - T[self.cam], R[self.cam])
        u, v = _project(self.intr[self.cam], Xc)
        return torch.stack([u, v], 1) - self.uv, Xc

    def cost(self, R, T, X):
        e, Xc = self.residual(R, T, X)
        s = (e * e).sum(1)
        rho = torch.where(s <= HUBER_PX ** 2, s, 2 * HUBER_PX * s.sqrt() - HUBER_PX ** 2)
        F = 0.5 * (rho * (Xc[:, 2] > 1e-6)).sum() / SIGMA_PX ** 2
        phi = _log3(self.Rp[self.free].transpose(1, 2) @ R[self.free])
        dT = T[self.free] - self.Tp[self.free]
        return F + 0.5 * (phi * phi).sum() / SIGMA_IMU ** 2 + 0.5 * (dT * dT).sum() / SIGMA_GNSS ** 2

    def jacobians(self):
        e, Xc = self.residual(self.R, self.T, self.X)
        f, _, _, k1, k2, p1, p2 = self.intr[self.cam].unbind(1)
        z = Xc[:, 2]
        a, b = Xc[:, 0] / z, Xc[:, 1] / z
        r2 = a * a + b * b
        rad, dr = 1 + r2 * (k1 + k2 * r2), 2 * k1 + 4 * k2 * r2
        s = (e * e).sum(1)
        scale = torch.where(s <= HUBER_PX ** 2, torch.ones_like(s), (HUBER_PX / s.sqrt()).sqrt()) / SIGMA_PX
        D00 = rad + dr * a * a + 2 * p1 * b + 6 * p2 * a
        D01 = dr * a * b + 2 * p1 * a + 2 * p2 * b
        D11 = rad + dr * b * b + 6 * p1 * b + 2 * p2 * a
        A = torch.stack([D00, D01, -(D00 * a + D01 * b), D01, D11, -(D01 * a + D11 * b)], 1).reshape(-1, 2, 3)
        A = A * (scale * f / z)[:, None, None]
        Jp = A @ self.R[self.cam].transpose(1, 2)
        return e * scale[:, None], torch.cat([A @ _hat(Xc), -Jp], 2), Jp

    def step(self, mu):
        r, Jc, Jp = self.jacobians()
        nf, free = self.nf, self.fi[self.cam] >= 0
        fc = self.fi[self.cam][free]
        zeros = lambda *n: torch.zeros(*n, dtype=torch.float64, device="cuda")  # noqa: E731
        Jf, rf = Jc[free], r[free]
        U = zeros(nf, 6, 6).index_add_(0, fc, Jf.transpose(1, 2) @ Jf)
        gc = zeros(nf, 6).index_add_(0, fc, -torch.einsum("nri,nr->ni", Jf, rf))
        V = zeros(self.np, 3, 3).index_add_(0, self.pt, Jp.transpose(1, 2) @ Jp)
        gp = zeros(self.np, 3).index_add_(0, self.pt, -torch.einsum("nri,nr->ni", Jp, r))
        phi = _log3(self.Rp[self.free].transpose(1, 2) @ self.R[self.free])
        t = phi.norm(dim=1)
        c2 = torch.where(t < 1e-3, 1 / 12 + t * t / 720,
                         1 / t.clamp(min=1e-9) ** 2 - (1 + t.cos()) / (2 * t * t.sin()).clamp(min=1e-18))
        K = _hat(phi)
        Jr = torch.eye(3, dtype=torch.float64, device="cuda") + 0.5 * K + c2[:, None, None] * (K @ K)
        U[:, :3, :3] += Jr.transpose(1, 2) @ Jr / SIGMA_IMU ** 2
        gc[:, :3] -= torch.einsum("nri,nr->ni", Jr, phi) / SIGMA_IMU ** 2
        U[:, 3:, 3:] += torch.eye(3, dtype=torch.float64, device="cuda") / SIGMA_GNSS ** 2
        gc[:, 3:] -= (self.T[self.free] - self.Tp[self.free]) / SIGMA_GNSS ** 2
        Dc = U.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32).clone()
        Dp = V.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32).clone()
        Vi = torch.linalg.inv(V + mu * torch.diag_embed(Dp))
        W = Jc.transpose(1, 2) @ Jp  # 6 x 3 of each observation
        Y = W @ Vi[self.pt]
        Wf, Yf, pf = W[free], Y[free], self.pt[free]
        S = zeros(nf * nf, 6, 6)
        diag = torch.arange(nf, device="cuda") * (nf + 1)
        S[diag] = U + mu * torch.diag_embed(Dc)
        S.index_add_(0, fc * (nf + 1), Yf @ Wf.transpose(1, 2), alpha=-1)
        rhs = gc - zeros(nf, 6).index_add_(0, fc, torch.einsum("nij,nj->ni", Yf, gp[pf]))
        for i in range(0, len(self.pair[0]) if self.pair else 0, 1 << 21):
            a, b = self.pair[0][i:i + (1 << 21)], self.pair[1][i:i + (1 << 21)]
            fa, fb = self.fi[self.cam[a]], self.fi[self.cam[b]]
            B = Y[a] @ W[b].transpose(1, 2)
            S.index_add_(0, fa * nf + fb, B, alpha=-1)
            S.index_add_(0, fb * nf + fa, B.transpose(1, 2).contiguous(), alpha=-1)
        M = S.reshape(nf, nf, 6, 6).transpose(1, 2).reshape(6 * nf, 6 * nf)
        dc = torch.linalg.solve(M, rhs.reshape(-1, 1)).reshape(nf, 6)
        back = zeros(self.np, 3).index_add_(0, pf, torch.einsum("nij,ni->nj", Wf, dc[fc]))
        dX = torch.einsum("nij,nj->ni", Vi, gp - back)
        pred = 0.5 * ((dc * (mu * Dc * dc + gc)).sum() + (dX * (mu * Dp * dX + gp)).sum())
        R, T = self.R.clone(), self.T.clone()
        R[self.free] = self.R[self.free] @ _exp(dc[:, :3])
        T[self.free] = self.T[self.free] + dc[:, 3:]
        return R, T, self.X + dX, float(pred)

    def solve(self, iters):
        mu, nu, F = MU0, 2.0, float(self.cost(self.R, self.T, self.X))
        for _ in range(iters):
            R, T, X, pred = self.step(mu)
            Fn = float(self.cost(R, T, X))
            gain = (F - Fn) / pred if pred > 0 else 0.0
            if gain > 0:
                self.R, self.T, self.X, F = R, T, X, Fn
                mu, nu = mu * max(1 / 3, 1 - (2 * gain - 1) ** 3), 2.0
            else:
                mu, nu = mu * nu, 2 * nu
        return F


def exact(case, seed):
    kind = case["kind"]
    if kind == "formation":
        return _formation_exact(case, seed)
    if kind == "cost":
        sc = _scene(seed, case["strips"], case["images"], case["points"], "all", 2, device_arrays=True)
        P = _Problem(sc)
        return P.cost(P.R, P.T, P.X).reshape(1)
    if case.get("clusters", 0) > 24:
        return None  # minutes in 64 bits
    Rs, Ts, Xs, Fs = [], [], [], []
    for sc in _scenes(case, seed):
        P = _Problem(sc)
        Fs.append(P.solve(case["iters"]))
        Rs.append(P.R.reshape(-1, 9))
        Ts.append(P.T)
        Xs.append(P.X)
    out = [torch.cat(Rs), torch.cat(Ts), torch.cat(Xs)]
    if kind == "window":
        out.append(P.residual(P.R, P.T, P.X)[0].norm(dim=1))
    elif kind != "run":
        out.append(np.array(Fs))
    return out


def _clip_area(A, B):
    """Area of the intersection of two convex quadrilaterals."""
    sign = 1.0 if sum(B[i][0] * B[(i + 1) % 4][1] - B[(i + 1) % 4][0] * B[i][1] for i in range(4)) >= 0 else -1.0
    P = A
    for e in range(4):
        (ex, ey), (fx, fy) = B[e], B[(e + 1) % 4]
        side = [sign * ((fx - ex) * (y - ey) - (fy - ey) * (x - ex)) for x, y in P]
        Q = []
        for i, (x, y) in enumerate(P):
            j = (i + 1) % len(P)
            if side[i] >= 0:
                Q.append((x, y))
            if (side[i] >= 0) != (side[j] >= 0):
                w = side[i] / (side[i] - side[j])
                Q.append((x + w * (P[j][0] - x), y + w * (P[j][1] - y)))
        P = Q
        if len(P) < 3:
            return 0.0
    return abs(0.5 * sum(P[i][0] * P[(i + 1) % len(P)][1] - P[(i + 1) % len(P)][0] * P[i][1] for i in range(len(P))))


def _formation_exact(case, seed):
    f = _formation_inputs(case, seed)
    n, dsm = len(f["R"]), f["dsm"]
    R, T, K, h = f["R"].reshape(n, 3, 3), f["T"], f["intr"], dsm["h"]
    ny, nx = h.shape

    def height(x, y):
        fx = np.clip((x - dsm["x0"]) / dsm["dx"], 0.0, nx - 1.0)
        fy = np.clip((y - dsm["y0"]) / dsm["dy"], 0.0, ny - 1.0)
        ix, iy = np.minimum(fx.astype(int), nx - 2), np.minimum(fy.astype(int), ny - 2)
        ax, ay = fx - ix, fy - iy
        return (h[iy, ix] * (1 - ax) + h[iy, ix + 1] * ax) * (1 - ay) + (h[iy + 1, ix] * (1 - ax) + h[iy + 1, ix + 1] * ax) * ay

    px = np.array([[0.0, 0.0], [WIDTH, 0.0], [WIDTH, HEIGHT], [0.0, HEIGHT]])
    ray = np.concatenate([(px[None] - K[:, None, 1:3]) / K[:, None, :1], np.ones((n, 4, 1))], 2)
    d = np.einsum("nij,ncj->nci", R, ray).reshape(-1, 3)
    o = np.repeat(T, 4, axis=0)
    above = lambda t: o[:, 2] + t * d[:, 2] - height(o[:, 0] + t * d[:, 0], o[:, 1] + t * d[:, 1])  # noqa: E731
    t0, t1 = np.maximum((o[:, 2] - h.max()) / -d[:, 2], 0.0), (o[:, 2] - h.min()) / -d[:, 2]
    m = np.maximum(np.ceil((t1 - t0) * np.hypot(d[:, 0], d[:, 1]) / (0.5 * dsm["dx"])), 1.0)
    lo, hi, found = t0.copy(), t1.copy(), np.zeros(len(o), dtype=bool)
    for i in range(1, int(m.max()) + 1):
        t = t0 + (t1 - t0) * i / m
        hit = ~found & (i <= m) & (above(t) <= 0)
        hi[hit], lo[hit] = t[hit], (t0 + (t1 - t0) * (i - 1) / m)[hit]
        found |= hit
    for _ in range(60):
        t = 0.5 * (lo + hi)
        under = above(t) <= 0
        hi, lo = np.where(under, t, hi), np.where(under, lo, t)
    corners = (o + hi[:, None] * d).reshape(n, 4, 3)
    quads = [[tuple(p[:2]) for p in c] for c in corners.tolist()]
    area = np.array([[_clip_area(a, b) for b in quads] for a in quads])
    q, m = f["p0"], slice(1, 1 + case["targets"])
    P = np.concatenate([(q - K[0, 1:3]) / K[0, 0], np.ones((len(q), 1))], 1)
    X = T[0] + f["depth"] * (P @ R[0].T)
    Xc = np.einsum("mni,mij->mnj", X[None] - T[m][:, None], R[m])
    p = K[m][:, None, :1] * Xc[..., :2] / Xc[..., 2:] + K[m][:, None, 1:3]
    return [corners, area, p, None]

"""Performance cases of the voxel-grid library: what a user has it do.

A case is a camera, a local grid and a form in which frames reach it.  Every
pass goes through the public binding (paper_2112_13169_gb300.vg) as a
robot's program does, one frame after another: integrate the measurement,
re-centre the grid on the robot, read the grid out for the planner.  Scenes
are seeded: boxes, spheres and cylinders in a room, ray-cast on the GPU,
with invalid pixels and depth noise; the robot moves about a voxel or more
between frames, with a heading drawn from the seed.

Outputs are the grids (voxel codes, bytes) and their origins (integers): they
have no rounding, so there is no value in 64 bits to compare them with.
"""
import math
import random

import numpy as np
import torch

from paper_2112_13169_gb300 import vg

# camera optical axes (x right, y down, z forward) in a forward-left-up body
BODY_CAM = np.array([[0.0, 0.0, 1.0], [-1.0, 0.0, 0.0], [0.0, -1.0, 0.0]])


def _case(name, form="grid", w=640, h=480, dtype="f32", fx=87.0, fy=58.0, depth=5.0, vs=0.05, nx=200, ny=200, nz=100,
          inf=2, frames=4, move=True, host=False, prims=200, points=0, count=1):
    c = dict(form=form, w=w, h=h, dtype=dtype, fx=fx, fy=fy, depth=depth, vs=vs, nx=nx, ny=ny, nz=nz, inf=inf,
             frames=frames, move=move, host=host, prims=prims, points=points, count=count)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one small frame into a small grid that does not
        # move (a robot hovering in a room), then the read; launches count
        _case("room", w=320, h=240, depth=4.0, vs=0.1, nx=80, ny=80, nz=40, inf=1, frames=1, move=False, prims=30),
        # the paper's own set-up: its camera, range, grid and inflation
        _case("paper", w=320, h=240, fx=85.0, fy=101.0, depth=6.5, vs=0.15, nx=100, ny=100, nz=20, prims=40),
        # an ordinary depth camera on an exploring robot; grid read in place
        # on the device (a planner on the GPU)
        _case("seq"),
        # the same with frames coming from page-locked host memory and the
        # grid going back there: a planner on the host
        _case("seq_host", host=True),
        # a high-resolution 16-bit depth camera with a large grid
        _case("hires_u16", w=1280, h=720, dtype="u16", fx=90.0, fy=60.0, depth=6.0, nx=400, ny=400, nz=120, frames=3,
              prims=600),
        # odd and ragged sizes all the way: image rows, grid rows, slices
        _case("ragged_u16", w=423, h=317, dtype="u16", fx=74.0, fy=61.0, depth=4.7, vs=0.06, nx=211, ny=173, nz=61,
              inf=3, prims=120),
        # a dense point cloud instead of an image (stereo, lidar), the
        # paper's grid; the count is odd
        _case("cloud_300k", form="points", points=299993, w=640, h=480, fx=85.0, fy=101.0, depth=6.5, vs=0.15, nx=100,
              ny=100, nz=20, prims=40),
        # a larger robot: inflation by 0.4 m
        _case("inflate_8", inf=8, frames=2),
        # fine mapping, the largest single grid: 2 cm voxels, long rays
        _case("fine", w=848, h=480, vs=0.02, nx=500, ny=500, nz=150, inf=5, frames=2),
        # a fleet in one fused launch, resolutions and grids mixed; four
        # steps, then every grid is read
        _case("batch_64", form="batch", count=64, prims=80),
        # a small fleet, a step and a read of every grid
        _case("batch_8", form="batch", count=8, frames=1, prims=80),
        # cameras of every kind served from pageable host memory: a burst of
        # two frames each, waited for, then every grid is read
        _case("served_12", form="served", count=12, frames=2, prims=80),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.random()
    if kind < 0.1:
        return _case(None, form="batch", count=_log(rng, 2, 64), frames=rng.randint(1, 4), prims=80,
                     inf=rng.randint(0, 3))
    if kind < 0.15:
        return _case(None, form="served", count=rng.randint(2, 12), frames=rng.randint(1, 2), prims=80)
    while True:
        vs = round(math.exp(rng.uniform(math.log(0.02), math.log(0.2))), 3)
        c = _case(None, w=_log(rng, 160, 1280), h=_log(rng, 120, 720), dtype=rng.choice(["f32", "u16"]),
                  fx=round(rng.uniform(50.0, 100.0), 1), fy=round(rng.uniform(40.0, 101.0), 1),
                  depth=round(rng.uniform(3.0, 7.0), 2), vs=vs, nx=_log(rng, 60, 500), ny=_log(rng, 60, 500),
                  nz=_log(rng, 20, 150), inf=rng.choice([0, 1, 1, 2, 2, 2, 3, 3, 5, 8]), frames=rng.randint(1, 4),
                  move=rng.random() < 0.9, host=rng.random() < 0.2, prims=_log(rng, 30, 300))
        if kind > 0.85:
            c["form"], c["points"], c["host"] = "points", _log(rng, 1000, 300000), False
        # no more rays and voxels than the largest listed case
        vd, hw, hh = _bundle(c)
        if c["frames"] * (2 * hw + 1) * (2 * hh + 1) * vd <= 2 * 475 * 279 * 250 and vd >= 20:
            return c


def _bundle(c):
    vd = round(c["depth"] / c["vs"])
    return vd, round(math.tan(math.radians(c["fx"] / 2)) * vd), round(math.tan(math.radians(c["fy"] / 2)) * vd)


def _members(case):
    """The cameras and grids of a case: itself, or a mixed fleet."""
    if case["form"] == "batch":
        r = random.Random(7)   # the mix is the case's, the scenes are the seed's
        out = []
        for _ in range(case["count"]):
            w, h = r.choice([(320, 240), (640, 480), (848, 480)])
            out.append(dict(case, w=w, h=h, vs=r.choice([0.05, 0.1, 0.2]), nx=r.randint(80, 256), ny=r.randint(80, 256),
                            nz=r.randint(40, 96), inf=r.randint(1, 3) if case["inf"] else 0))
        return out
    if case["form"] == "served":
        small = dict(w=320, h=240, vs=0.1, nx=80, ny=80, nz=40, inf=1, depth=4.0)
        large = dict(w=1280, h=720, vs=0.05, nx=400, ny=400, nz=120, depth=6.0, fx=90.0, fy=60.0)
        kinds = [small, {}, dict(dtype="u16"), dict(large, dtype="u16"), dict(small, dtype="u16"), large]
        return [dict(case, **kinds[k % 6]) for k in range(case["count"])]
    return [case]


def work(case):
    """Each frame is read once; each grid is read and written once for every
    read-out.  Operations: about 40 a pixel or point, 16 a voxel of a ray."""
    nbytes = flops = 0
    for m in _members(case):
        vd, hw, hh = _bundle(m)
        n = m["nx"] * m["ny"] * m["nz"]
        px = m["points"] or m["w"] * m["h"]
        reads = m["frames"] if m["form"] in ("grid", "points") else 1
        nbytes += m["frames"] * px * (12 if m["points"] else 4 if m["dtype"] == "f32" else 2) + 2 * n * reads
        steps = min(vd + (hw + hh) / 2, (m["nx"] + m["ny"] + m["nz"]) / 2)
        flops += m["frames"] * (40 * px + 16 * (2 * hw + 1) * (2 * hh + 1) * steps)
    return {"bytes": float(nbytes), "flops": float(flops)}


def exact(case, seed):
    return None   # voxel codes and origins are whole numbers


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
def _pose(pos, yaw, pitch, roll):
    cy, sy, cp, sp, cr, sr = math.cos(yaw), math.sin(yaw), math.cos(pitch), math.sin(pitch), math.cos(roll), math.sin(roll)
    rz = np.array([[cy, -sy, 0], [sy, cy, 0], [0, 0, 1.0]])
    ry = np.array([[cp, 0, sp], [0, 1.0, 0], [-sp, 0, cp]])
    rx = np.array([[1.0, 0, 0], [0, cr, -sr], [0, sr, cr]])
    T = np.eye(4)
    T[:3, :3] = rz @ ry @ rx @ BODY_CAM
    T[:3, 3] = pos
    return T


def _scene(rng, m, path):
    """Boxes, spheres and cylinders in a room around the path, none near it."""
    half = max(1.5 * m["depth"], 0.5 * m["vs"] * max(m["nx"], m["ny"]))
    hi = np.array([half, half, 2.5])
    lo = np.array([-half, -half, -1.5])
    boxes, spheres, cyls = [], [], []
    while len(boxes) + len(spheres) + len(cyls) < m["prims"]:
        c, kind = rng.uniform(lo, hi), rng.integers(3)
        s = rng.uniform(0.1, 0.6, 3)
        gap = np.abs(path - c)
        if (np.all(gap < s.max() + 0.5, axis=1) if kind < 2 else np.all(gap[:, :2] < s[0] + 0.5, axis=1)).any():
            continue
        if kind == 0:
            boxes.append(np.concatenate([c - s, c + s]))
        elif kind == 1:
            spheres.append([c[0], c[1], c[2], s[0]])
        else:
            cyls.append([c[0], c[1], lo[2], min(hi[2], lo[2] + rng.uniform(0.5, 4.0)), s[0]])
    room = np.concatenate([lo, hi])
    return [torch.tensor(np.array(v, np.float32).reshape(-1, k), device="cuda")
            for v, k in ((boxes, 6), (spheres, 4), (cyls, 5), (room, 6))]


def _render(scene, T, m):
    """z-depth of every pixel (metres; the room encloses the camera)."""
    boxes, spheres, cyls, room = scene
    w, h = m["w"], m["h"]
    fx, fy = w / 2 / math.tan(math.radians(m["fx"] / 2)), h / 2 / math.tan(math.radians(m["fy"] / 2))
    u = (torch.arange(w, device="cuda", dtype=torch.float32) - (w - 1) / 2) / fx
    v = (torch.arange(h, device="cuda", dtype=torch.float32) - (h - 1) / 2) / fy
    R = torch.tensor(T[:3, :3].astype(np.float32), device="cuda")
    o = torch.tensor(T[:3, 3].astype(np.float32), device="cuda")
    d = (R[:, 0, None, None] * u[None, None, :] + R[:, 1, None, None] * v[None, :, None] + R[:, 2, None, None])
    d = torch.where(d.abs() < 1e-6, torch.full_like(d, 1e-6), d).reshape(3, 1, h * w)
    inv = 1.0 / d
    best = torch.full((h * w,), math.inf, device="cuda")

    def slabs(b):
        near = torch.full((len(b), h * w), -math.inf, device="cuda")
        far = torch.full((len(b), h * w), math.inf, device="cuda")
        for k in range(3):
            t0, t1 = (b[:, k, None] - o[k]) * inv[k], (b[:, 3 + k, None] - o[k]) * inv[k]
            near, far = torch.maximum(near, torch.minimum(t0, t1)), torch.minimum(far, torch.maximum(t0, t1))
        return near, far

    best = torch.minimum(best, slabs(room)[1][0])
    for b in boxes.split(32):
        near, far = slabs(b)
        best = torch.minimum(best, torch.where((near < far) & (near > 0), near, math.inf).amin(0))
    for s in spheres.split(32):
        q = o[:, None, None] - s[:, :3].T[:, :, None]
        aa, bb, cc = (d * d).sum(0), (d * q).sum(0), (q * q).sum(0) - s[:, 3, None] ** 2
        disc = bb * bb - aa * cc
        t = (-bb - disc.clamp_min(0).sqrt()) / aa
        best = torch.minimum(best, torch.where((disc > 0) & (t > 0), t, math.inf).amin(0))
    for s in cyls.split(32):
        q = o[:2, None, None] - s[:, :2].T[:, :, None]
        aa, bb = (d[:2] * d[:2]).sum(0), (d[:2] * q).sum(0)
        disc = bb * bb - aa * ((q * q).sum(0) - s[:, 4, None] ** 2)
        t = (-bb - disc.clamp_min(0).sqrt()) / aa
        z = o[2] + t * d[2]
        best = torch.minimum(best, torch.where((disc > 0) & (t > 0) & (z > s[:, 2, None]) & (z < s[:, 3, None]), t, math.inf).amin(0))
    return best.reshape(h, w)


def _frames(m, seed, member):
    """[(input, pose, robot position)] of one camera: depth images or clouds."""
    rng = np.random.default_rng([seed, member])
    g = torch.Generator(device="cuda").manual_seed(seed * 1009 + member)
    yaw = rng.uniform(-math.pi, math.pi)
    step = max(0.05, 1.2 * m["vs"]) if m["move"] else 0.0
    tilt = 0.03 if m["move"] else 0.0
    path = np.array([[math.cos(yaw) * step * i, math.sin(yaw) * step * i, 0.2 * step * i] for i in range(m["frames"])])
    path += rng.uniform(-0.5, 0.5, 3) * (1.0, 1.0, 0.2)
    scene = _scene(rng, m, path)
    out = []
    for p in path:
        T = _pose(p, yaw + rng.uniform(-tilt, tilt), rng.uniform(-tilt, tilt), rng.uniform(-tilt, tilt))
        d = _render(scene, T, m)
        d = d * (1.0 + 0.01 * torch.randn(d.shape, generator=g, device="cuda"))
        if m["points"]:
            # the cloud: points of the image's surfaces between the pixels
            h, w = d.shape
            px = torch.randint(h * w, (m["points"],), generator=g, device="cuda")
            z = d.reshape(-1)[px]
            x = ((px % w) - (w - 1) / 2) * z / (w / 2 / math.tan(math.radians(m["fx"] / 2)))
            y = (torch.div(px, w, rounding_mode="floor") - (h - 1) / 2) * z / (h / 2 / math.tan(math.radians(m["fy"] / 2)))
            x = torch.stack([x, y, z], 1).contiguous()
        else:
            d = torch.where(torch.rand(d.shape, generator=g, device="cuda") < 0.1, torch.zeros_like(d), d)
            if m["dtype"] == "u16":
                d = (d * 1000.0).round().clamp(0, 65535).to(torch.int32).to(torch.uint16)
            x = d.contiguous()
        if m["host"]:
            x = x.cpu().pin_memory()
        elif m["form"] == "served":
            x = x.cpu().numpy()
        out.append((x, np.ascontiguousarray(T), p.copy()))
    return out


def prepare(case, seed):
    members = _members(case)
    frames = [_frames(m, seed, k) for k, m in enumerate(members)]
    scale = [0.001 if m["dtype"] == "u16" else 1.0 for m in members]
    sizes = [m["nx"] * m["ny"] * m["nz"] for m in members]
    at = np.concatenate([[0], np.cumsum([-(-n // 256) * 256 for n in sizes])])
    out = torch.zeros(int(at[-1]), dtype=torch.uint8, device="cpu" if case["host"] else "cuda")
    if case["host"]:
        out = out.pin_memory()
    st = {"case": case, "frames": frames, "scale": scale, "out": out,
          "views": [out[int(a):int(a) + n] for a, n in zip(at, sizes)]}
    if case["form"] == "served":
        st["server"] = vg.Server(4 << 30, max_batch=64)
        st["cams"] = [st["server"].add_camera((m["nx"], m["ny"], m["nz"]), m["vs"], m["fx"], m["fy"], m["depth"],
                                              m["inf"], f[0][2]) for m, f in zip(members, frames)]
    else:
        st["grids"] = [vg.Grid((m["nx"], m["ny"], m["nz"]), m["vs"], m["fx"], m["fy"], m["depth"], m["inf"], f[0][2])
                       for m, f in zip(members, frames)]
    if case["form"] == "batch":
        st["batch"] = vg.Batch(len(members))
    return st


def run(state):
    case, views = state["case"], state["views"]
    if case["form"] == "batch":
        grids = state["grids"]
        for k in range(case["frames"]):
            state["batch"].step([(g, f[k][0], f[k][1], f[k][2] if case["move"] else None, s)
                                 for g, f, s in zip(grids, state["frames"], state["scale"])])
        origins = [g.read(v) for g, v in zip(grids, views)]
    elif case["form"] == "served":
        server, cams = state["server"], state["cams"]
        tickets = [server.submit(c, f[k][0], f[k][1], f[k][2], s)
                   for k in range(case["frames"]) for c, f, s in zip(cams, state["frames"], state["scale"])]
        for t in tickets:
            if server.wait(t) != vg.VG_OK:
                raise RuntimeError("a served frame failed")
        origins = [server.read(c, v) for c, v in zip(cams, views)]
    else:
        grid, scale = state["grids"][0], state["scale"][0]
        for x, T, pos in state["frames"][0]:
            if case["form"] == "points":
                grid.integrate_points(x, T)
            else:
                grid.integrate_depth(x, T, scale)
            if case["move"]:
                grid.shift(pos)
            origins = [grid.read(views[0])]
    return {"grid": state["out"], "origin": np.array(origins)}

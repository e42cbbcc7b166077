"""Performance cases: what a user of the renderer has it do, from a small training step to a
loss over full-HD views of a 1024^3 cube, through the package's public calls.

Sizes come from the benchmark's workloads and the tests (128^3 at 256^2, 512^3 at 1024^2,
1024^3 at 1920x1080, batches of uneven cubes, rays 6 voxels apart in a large cube, the small
ragged cubes of the tests); `draw` spreads them over the ranges in between.  Cubes are
noise with Gaussian sources (the structure of a 21-cm spectral cube), tables the benchmark's
ramp (transparent below two standard deviations of the noise) or random piecewise linear ones.

`exact` computes the same outputs in 64 bits with plain torch operations."""
import math
import random

import torch

import paper_1211_4896_gb300 as P
from paper_1211_4896_gb300.sortlast import split_cells

VMIN, VMAX, K, FOV = -3.0, 50.0, 256, 40.0
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------

def _case(kind, dims, size, name=None, store="f32", views=1, step=1.0, ert=0.99, table="ramp", proj="persp", az=0.0,
          el=0.0, **more):
    c = dict(kind=kind, nx=dims[0], ny=dims[1], nz=dims[2], w=size[0], h=size[1], store=store, views=views, step=step,
             ert=ert, table=table, proj=proj, az=az, el=el, **more)
    return dict(name=name, **c) if name else c


def listed():
    big, hd = (1024, 1024, 1024), (1920, 1080)
    return [
        # a small cube seen whole, face on: one short launch
        _case("view", (128, 128, 128), (256, 256), "view_plain_128", step=0.5, ert=2.0, proj="ortho"),
        # one frame of an interactive view of a large cube, oblique
        _case("view", big, hd, "view_1080p", az=45.0),
        # a frame of a ragged cube kept in 16 bits, tilted
        _case("view", (705, 611, 833), (1000, 750), "view_half", store="f16", az=30.0, el=20.0),
        # a preview of a cube with many more voxels than the image has pixels: rays 6 voxels apart
        _case("view", (2048, 2048, 1024), (960, 540), "view_sparse", az=45.0),
        # thumbnails of many uneven cubes in one call
        _case("batch", (512, 512, 1024), (1024, 1024), "batch_uneven", store="f16", views=16, table="pwl", sizes=4),
        # one step of fitting a table and a cube to views of a large cube: forward and backward, full HD
        _case("fit", big, hd, "step_1024", views=2, az=10.0, batched=True),
        # the same where each voxel takes several samples: dense views, fine step, no early end
        _case("fit", (512, 512, 512), (1024, 1024), "grad_512", views=4, step=0.5, ert=2.0, table="pwl", az=20.0,
              batched=False),
        # the smallest training step: new voxels, forward, loss, backward through autograd
        _case("train", (44, 36, 40), (61, 47), "train_small", step=0.5, az=15.0, el=10.0),
        # what a viewer asks once a cube is loaded: moments, histogram over the data range, exact median
        _case("stats", big, (1, 1), "stats_1024"),
        # sigma clipping: statistics of 32^3 regions and the view that uses them
        _case("sigma", (640, 720, 500), (1280, 720), "sigma_view", az=70.0, el=-10.0, region=32),
        # maximum intensity projection along a cube's x axis
        _case("mip", big, hd, "mip_1080p", ert=2.0, az=90.0),
        # sort-last: the partial images of eight sub-boxes and their composite
        _case("sortlast", big, hd, "sortlast_8", ert=2.0, az=20.0, boxes=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "view", "batch", "fit", "train", "stats", "sigma", "mip", "sortlast"])
    while True:
        top = 160 if kind == "train" else (2048 if kind == "view" else 1100)
        dims = [_log_int(rng, 36, top) for _ in range(3)]
        h = _log_int(rng, 45, 1080)
        size = [max(45, round(h * rng.uniform(0.9, 1.8))), h]
        step = rng.choice([0.5, 0.7, 1.0, 1.0])
        c = _case(kind, dims, size, store=rng.choice(["f32", "f32", "f16", "bf16"]), step=step,
                  ert=rng.choice([0.99, 0.99, 2.0]), table=rng.choice(["ramp", "ramp", "pwl"]),
                  proj=rng.choice(["persp", "persp", "ortho"]), az=round(rng.uniform(0.0, 360.0), 1),
                  el=round(rng.uniform(-35.0, 35.0), 1))
        if kind == "batch":
            c.update(views=rng.randint(2, 16), sizes=rng.randint(0, 1 << 20))
        elif kind == "fit":
            c.update(views=rng.randint(1, 4), batched=rng.random() < 0.5, store="f32")
        elif kind == "train":
            c.update(store="f32")
        elif kind == "stats":
            c.update(w=1, h=1)
        elif kind == "sigma":
            c.update(region=rng.randint(8, 64), ert=0.99)
        elif kind == "mip":
            c.update(ert=2.0)
        elif kind == "sortlast":
            c.update(boxes=rng.choice([2, 3, 4, 6, 8]), ert=2.0)
        if math.prod(dims) <= 1 << 32 and (kind == "stats" or _cost(c) <= 1.0e9):
            return c


# ------------------------------------------------------------------------------------------
# Geometry, cameras, tables, cubes
# ------------------------------------------------------------------------------------------

def _camera(dims, w, h, proj, az, el):
    """A view of the cube's centre from azimuth az and elevation el (degrees) whose height fits the bounding sphere."""
    centre = [(d - 1) / 2.0 for d in dims]
    radius = 0.5 * math.sqrt(sum((d - 1) ** 2 for d in dims))
    a, e = math.radians(az), math.radians(el)
    f = (-math.cos(e) * math.sin(a), -math.sin(e), math.cos(e) * math.cos(a))
    dist = radius / math.sin(math.radians(FOV) / 2.0)
    if proj == "ortho":          # the height of the box as it stands, seen face on
        return dict(kind=P.VR_CAMERA_ORTHO, eye=tuple(c - 2.0 * radius * x for c, x in zip(centre, f)), forward=f,
                    up=(0.0, 1.0, 0.0), fov_y_deg=0.0, ortho_height=float(dims[1] - 1), width=w, height=h)
    return dict(kind=P.VR_CAMERA_PERSPECTIVE, eye=tuple(c - dist * x for c, x in zip(centre, f)), forward=f,
                up=(0.0, 1.0, 0.0), fov_y_deg=FOV, ortho_height=0.0, width=w, height=h)


def _pitch(dims, c):
    """Distance of neighbouring rays at the cube's centre, in voxels."""
    if c["proj"] == "ortho":
        return (dims[1] - 1) / c["h"]
    return math.sqrt(sum((d - 1) ** 2 for d in dims)) / math.cos(math.radians(FOV) / 2.0) / c["h"]


def _jobs(case):
    """(dims, camera) of every view of a case."""
    if case["kind"] == "batch":
        r, out = random.Random(case["sizes"]), []
        for _ in range(case["views"]):
            d = [r.randrange(64, n + 1, 32) if n >= 64 else n for n in (case["nx"], case["ny"], case["nz"])]
            s = r.randint(max(1, case["w"] // 2), case["w"]), r.randint(max(1, case["h"] // 2), case["h"])
            out.append((d, _camera(d, s[0], s[1], case["proj"], r.uniform(0.0, 360.0), r.uniform(-35.0, 35.0))))
        return out
    d = (case["nx"], case["ny"], case["nz"])
    return [(d, _camera(d, case["w"], case["h"], case["proj"], case["az"] + 90.0 * v, case["el"]))
            for v in range(case["views"])]


def _samples(dims, cam, c):
    """About how many samples a view takes: the cube's volume over the volume of one sample (in the image's frame)."""
    pitch = _pitch(dims, dict(c, h=cam["height"]))
    inside = min(1.0, (cam["width"] * pitch) / max(dims))            # narrow images cut the cube off
    return max(1.0, math.prod(dims) * inside / (pitch * pitch * c["step"]))


def _cost(case):
    per = 3.0 if case["kind"] in ("fit", "train") else 1.0
    return per * sum(_samples(d, cam, case) for d, cam in _jobs(case)) + 0.2 * math.prod(_jobs(case)[0][0])


def work(case):
    """Voxels that the rays' trilinear footprints touch, once for each call that reads them, plus the images; two
    thirds of the operations of a sample are its interpolation."""
    size = 4 if case["store"] == "f32" else 2
    nvox = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "stats":
        return {"bytes": float(nvox * size), "flops": 8.0 * nvox}
    total, flops = 0.0, 0.0
    seen = 0.0
    for d, cam in _jobs(case):
        n, px, v = _samples(d, cam, case), cam["width"] * cam["height"], math.prod(d)
        touched = min(v, 4.0 * n)                        # two by two voxel columns a ray
        seen = max(seen, touched)
        flops += 40.0 * n
        total += px * 20.0 + (touched * size if case["kind"] == "batch" else 0.0)
        if case["kind"] in ("fit", "train"):             # the image's gradient in; the march again, with its adjoint
            total += px * 16.0
            flops += 80.0 * n
    if case["kind"] != "batch":
        total += seen * size
    if case["kind"] in ("fit", "train"):
        total += nvox * 4.0                              # the voxels' gradient
    if case["kind"] == "sigma":
        total += max(0.0, nvox - seen) * size
        flops += 4.0 * nvox
    if case["kind"] == "sortlast":
        total += case["w"] * case["h"] * 20.0 * case["boxes"]
    return {"bytes": total, "flops": flops}


def _table(case, seed, device):
    """(K, 4) float32 RGBA: the linear ramp, transparent below the value 2, or 4 to 8 random knots a channel."""
    t = torch.linspace(0.0, 1.0, K, dtype=torch.float64)
    if case["table"] == "ramp":
        lo = 2.0 if case["kind"] != "sigma" else 8.0 * (2.0 - VMIN) / (VMAX - VMIN)
        top = VMAX if case["kind"] != "sigma" else 8.0
        v = t * (top - (VMIN if case["kind"] != "sigma" else 0.0)) + (VMIN if case["kind"] != "sigma" else 0.0)
        a = torch.where(v < lo, torch.zeros_like(v), 0.1 * (v - lo) / (top - lo))
        out = torch.stack([t, t * t, 1.0 - t, a], 1)
    else:
        r = random.Random(seed)
        n = r.randint(4, 8)
        x = torch.linspace(0.0, 1.0, n, dtype=torch.float64)
        at = torch.clamp(torch.searchsorted(x, t, right=True) - 1, 0, n - 2)
        w = (t - x[at]) * (n - 1)
        cols = []
        for ch in range(4):
            y = torch.tensor([r.random() for _ in range(n)], dtype=torch.float64)
            if ch == 3:
                y *= 0.15
                y[0] = 0.0
            cols.append(y[at] * (1.0 - w) + y[at + 1] * w)
        out = torch.stack(cols, 1)
    return out.to(torch.float32).to(device).contiguous()


def _cube(dims, seed, dtype):
    """Unit noise with Gaussian sources of amplitude 5 to 50, at the benchmark's density (at most 2000)."""
    nx, ny, nz = dims
    g = torch.Generator(device="cuda").manual_seed(seed)
    cube = torch.randn((nz, ny, nx), generator=g, device="cuda", dtype=torch.float32)
    r = random.Random(seed)
    for _ in range(min(2000, max(3, round(20 * nx * ny * nz / 128 ** 3)))):
        amp, sig = r.uniform(5.0, 50.0), r.uniform(2.0, 8.0)
        at, axes = [], []
        for n in (nx, ny, nz):
            c = r.uniform(0.0, n - 1.0)
            a, b = max(0, int(c - 4.0 * sig)), min(n, int(c + 4.0 * sig) + 1)
            at.append(slice(a, b))
            axes.append(torch.exp((torch.arange(a, b, device="cuda") - c) ** 2 * (-0.5 / (sig * sig))))
        cube[at[2], at[1], at[0]] += (amp * axes[2])[:, None, None] * axes[1][None, :, None] * axes[0][None, None, :]
    return cube.to(dtype)


def _range(case):
    return (0.0, 8.0) if case["kind"] == "sigma" else (VMIN, VMAX)


def _goal(case, cam, seed):
    """An image to fit or a gradient image: smooth noise of unit size, the same on every call with this seed."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    return torch.rand((cam["height"], cam["width"], 4), generator=g, device="cuda", dtype=torch.float32)


# ------------------------------------------------------------------------------------------
# What is timed
# ------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind, jobs = case["kind"], _jobs(case)
    s = dict(case=case, tf=_table(case, seed, "cuda"), cams=[cam for _, cam in jobs])
    if kind == "batch":
        s["vols"] = [P.Volume(_cube(d, seed + q, DTYPES[case["store"]]), case["store"])
                     for q, (d, _) in enumerate(jobs)]
    else:
        cube = _cube(jobs[0][0], seed, DTYPES[case["store"]])
        s["vols"] = [P.Volume(cube, case["store"])] * len(jobs)
        if kind == "train":
            s["cube"] = cube.requires_grad_(True)
            s["tf"] = s["tf"].requires_grad_(True)
    if kind in ("fit", "train"):
        s["goals"] = [_goal(case, cam, seed + q) for q, cam in enumerate(s["cams"])]
    if kind in ("batch", "fit"):         # a frame loop draws into images that it keeps
        lo, hi = _range(case)
        s["jobs"] = [dict(vol=v, cam=cam, tf=s["tf"], vmin=lo, vmax=hi, step=case["step"], ert=case["ert"],
                          out=torch.empty((cam["height"], cam["width"], 4), device="cuda"),
                          nsamples=torch.empty((cam["height"], cam["width"]), device="cuda", dtype=torch.int32))
                     for v, cam in zip(s["vols"], s["cams"])]
    return s


def run(s):
    case, vol, cam, tf = s["case"], s["vols"][0], s["cams"][0], s["tf"]
    kind, step, ert = case["kind"], case["step"], case["ert"]
    lo, hi = _range(case)
    if kind == "view":
        return P.render(vol, cam, tf, lo, hi, step, ert)
    if kind == "batch":
        P.render_batched(s["jobs"])
        return [(j["out"], j["nsamples"]) for j in s["jobs"]]
    if kind == "fit":
        jobs = s["jobs"]
        if case["batched"]:
            P.render_batched(jobs)
        else:
            for j in jobs:
                P.render(vol, j["cam"], tf, lo, hi, step, ert, out=j["out"], nsamples=j["nsamples"])
        grads = [2.0 / g.numel() * (j["out"] - g) for j, g in zip(jobs, s["goals"])]
        gtf, gvox = P.render_backward_views(vol, s["cams"], tf, lo, hi, step, [j["out"] for j in jobs],
                                            [j["nsamples"] for j in jobs], grads, ert)
        # the gradients as an optimiser of the float32 table and cube takes them
        return dict(images=[(j["out"], j["nsamples"]) for j in jobs], table=gtf.to(tf.dtype), voxels=gvox)
    if kind == "train":
        vol.update(s["cube"].detach())
        img = P.render_diff(s["cube"], tf, vol, cam, lo, hi, step, ert)
        loss = ((img - s["goals"][0]) ** 2).mean()
        gvox, gtf = torch.autograd.grad(loss, [s["cube"], tf])
        return dict(loss=loss.detach(), image=img.detach(), table=gtf, voxels=gvox)
    if kind == "stats":
        m = P.moments(vol)
        return dict(moments=m, histogram=P.histogram(vol, m["min"], m["max"], 256), median=P.median(vol))
    if kind == "sigma":
        region = (case["region"],) * 3
        mm = P.minimap(vol, region)
        img, n = P.render(vol, cam, tf, lo, hi, step, ert, mode=P.VR_MODE_SIGMA, minimap=mm, region=region)
        return dict(minimap=mm, image=img, nsamples=n)
    if kind == "mip":
        return P.render(vol, cam, tf, lo, hi, step, ert, mode=P.VR_MODE_MIP)
    parts = [P.render_subbox(vol, cam, tf, lo, hi, step, a, b)
             for a, b in split_cells([n - 1 for n in vol.dims], case["boxes"])]
    image = P.composite([p[0] for p in parts], [p[1] for p in parts])
    return dict(image=image, parts=parts)


# ------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------

class _View:
    """One view's rays: samples sit at t_in + (k + 1/2) step, up to the far side of the box."""

    def __init__(self, dims, cam, step):
        f = torch.tensor(cam["forward"], dtype=torch.float64)
        f = f / f.norm()
        r = torch.linalg.cross(f, torch.tensor(cam["up"], dtype=torch.float64))
        r = r / r.norm()
        u = torch.linalg.cross(r, f)
        w, h = cam["width"], cam["height"]
        half = math.tan(math.radians(cam["fov_y_deg"]) / 2.0) if cam["kind"] == P.VR_CAMERA_PERSPECTIVE else \
            0.5 * cam["ortho_height"]
        x = ((torch.arange(w, dtype=torch.float64, device="cuda") + 0.5) * 2.0 / w - 1.0) * half * w / h
        y = (1.0 - (torch.arange(h, dtype=torch.float64, device="cuda") + 0.5) * 2.0 / h) * half
        plane = x[None, :, None] * r.cuda() + y[:, None, None] * u.cuda()
        eye = torch.tensor(cam["eye"], dtype=torch.float64, device="cuda")
        if cam["kind"] == P.VR_CAMERA_PERSPECTIVE:
            d = plane + f.cuda()
            self.d, self.o = d / d.norm(dim=2, keepdim=True), eye.expand_as(d)
            near = 0.0
        else:
            self.d, self.o = f.cuda().expand_as(plane), eye + plane
            near = -math.inf
        self.d, self.o = self.d.reshape(-1, 3), self.o.reshape(-1, 3)
        top = torch.tensor([n - 1.0 for n in dims], dtype=torch.float64, device="cuda")
        a, b = (0.0 - self.o) / self.d, (top - self.o) / self.d
        flat = self.d == 0.0
        out = flat & ((self.o < 0.0) | (self.o > top))
        a, b = torch.where(flat, -math.inf, a), torch.where(flat, math.inf, b)
        self.t = torch.clamp(torch.minimum(a, b).amax(1), min=near)
        far = torch.maximum(a, b).amin(1)
        n = torch.floor((far - self.t) / step + 0.5)
        self.n = torch.where(out.any(1) | ~(far > self.t), torch.zeros_like(n), n).long()
        self.step, self.size = step, (h, w)


class _Field:
    def __init__(self, cube, tf, lo, hi):
        self.v, (self.nz, self.ny, self.nx) = cube.reshape(-1), cube.shape
        self.tf, self.lo, self.scale = tf.detach().double(), lo, (K - 1) / (float(hi) - float(lo))

    def cell(self, p):
        n = torch.tensor([self.nx, self.ny, self.nz], device="cuda")
        c = torch.minimum(torch.clamp(torch.floor(p).long(), min=0), n - 2)
        w = p - c
        base = (c[:, 2] * self.ny + c[:, 1]) * self.nx + c[:, 0]
        return [base + dz * self.ny * self.nx + dy * self.nx + dx for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)], \
            [(w[:, 0] if dx else 1 - w[:, 0]) * (w[:, 1] if dy else 1 - w[:, 1]) * (w[:, 2] if dz else 1 - w[:, 2])
             for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)]

    def value(self, cell):
        return sum(w * self.v[i].double() for i, w in zip(*cell))

    def look_up(self, v):
        u = torch.clamp((v - self.lo) * self.scale, 0.0, K - 1.0)
        i = torch.clamp(u.long(), max=K - 2)
        w = (u - i)[:, None]
        return i, w, self.tf[i] * (1.0 - w) + self.tf[i + 1] * w


def _march(view, field, visit, n=None):
    """visit(rays, k, cell, value) for the k-th samples of the rays that have one and that visit has not ended (it
    returns those that go on)."""
    n = view.n if n is None else n
    live, k = torch.nonzero(n > 0)[:, 0], 0
    while live.numel():
        t = view.t[live] + (k + 0.5) * view.step
        cell = field.cell(view.o[live] + t[:, None] * view.d[live])
        on = visit(live, k, cell, field.value(cell))
        k += 1
        on = (n[live] > k) if on is None else on & (n[live] > k)
        live = live[on]


def _render64(view, field, ert, change=lambda rays, k, v: v):
    px = view.n.numel()
    c = torch.zeros((px, 3), dtype=torch.float64, device="cuda")
    t = torch.ones(px, dtype=torch.float64, device="cuda")
    used = torch.zeros(px, dtype=torch.long, device="cuda")

    def visit(rays, k, cell, v):
        e = field.look_up(change(rays, k, v))[2]
        before = t[rays]
        c[rays] += (before * e[:, 3])[:, None] * e[:, :3]
        t[rays] = after = before * (1.0 - e[:, 3])
        used[rays] = k + 1
        return 1.0 - after < ert

    _march(view, field, visit)
    return c, t, used


def _image(c, t, view):
    return torch.cat([c, 1.0 - t[:, None]], 1).reshape(*view.size, 4)


def _adjoint64(view, field, c, t, used, g, gtf, gvox):
    """Adds the gradients of sum(g * image) to the table's and the voxels' (images over no background)."""
    g = g.double().reshape(-1, 4)
    rest = (c * g[:, :3]).sum(1) - g[:, 3] * t
    through = torch.ones_like(t)

    def visit(rays, k, cell, v):
        i, w, e = field.look_up(v)
        gr, before = g[rays], through[rays]
        cg = (e[:, :3] * gr[:, :3]).sum(1)
        rest[rays] = after = rest[rays] - before * e[:, 3] * cg
        da = before * cg - after / (1.0 - e[:, 3])
        through[rays] = before * (1.0 - e[:, 3])
        de = torch.cat([(before * e[:, 3])[:, None] * gr[:, :3], da[:, None]], 1)
        gtf.index_add_(0, i, (1.0 - w) * de)
        gtf.index_add_(0, i + 1, w * de)
        u = (v - field.lo) * field.scale
        dv = ((field.tf[i + 1] - field.tf[i]) * de).sum(1) * field.scale
        dv = torch.where((u > 0.0) & (u < K - 1.0), dv, torch.zeros_like(dv))
        at = torch.nonzero(dv)[:, 0]
        for q, weight in zip(*cell):
            gvox.index_add_(0, q[at], (weight * dv)[at])

    _march(view, field, visit, used)


def _regions(cube, r):
    """Mean and standard deviation of the cube's r^3 regions, (mz, my, mx, 2)."""
    rows = []
    for z in range(0, cube.shape[0], r):
        s = cube[z:z + r].double()
        n1 = torch.ones_like(s[:1])
        def fold(x):
            for d in (1, 2):
                m = -(-x.shape[d] // r)
                pad = [0] * 6
                pad[2 * (2 - d) + 1] = m * r - x.shape[d]
                x = torch.nn.functional.pad(x, pad)
                x = x.reshape(*x.shape[:d], m, r, *x.shape[d + 1:]).sum(d + 1)
            return x.sum(0)
        n = fold(n1) * s.shape[0]
        mean = fold(s) / n
        wide = mean.repeat_interleave(r, 0)[:s.shape[1]].repeat_interleave(r, 1)[:, :s.shape[2]]
        rows.append(torch.stack([mean, torch.sqrt(fold((s - wide) ** 2) / n)], 2))
    return torch.stack(rows)


def _sigma_units(view, field, mm, r):
    """The change of a sample's value into units of the regions' statistics around it."""
    m = torch.tensor([mm.shape[2], mm.shape[1], mm.shape[0]], device="cuda")

    def change(rays, k, v):
        p = view.o[rays] + (view.t[rays] + (k + 0.5) * view.step)[:, None] * view.d[rays]
        g = (p + 0.5) / r - 0.5
        i = torch.clamp(torch.minimum(torch.floor(g).long(), m - 2), min=0)
        w = torch.where(m > 1, torch.clamp(g - i, 0.0, 1.0), 0.0)
        j = torch.minimum(i + 1, m - 1)
        st = 0.0
        for q in range(8):
            at = [(j if q >> a & 1 else i)[:, a] for a in range(3)]
            wt = math.prod((w if q >> a & 1 else 1.0 - w)[:, a] for a in range(3))
            st = st + wt[:, None] * mm[at[2], at[1], at[0]]
        return (v - st[:, 0]) / torch.clamp(st[:, 1], min=1e-30)

    return change


def exact(case, seed):
    kind, jobs, (lo, hi) = case["kind"], _jobs(case), _range(case)
    tf, step, ert = _table(case, seed, "cuda"), case["step"], case["ert"]
    if kind == "batch":
        out = []
        for q, (d, cam) in enumerate(jobs):
            view, field = _View(d, cam, step), _Field(_cube(d, seed + q, DTYPES[case["store"]]), tf, lo, hi)
            out.append((_image(*_render64(view, field, ert)[:2], view), None))
        return out
    cube = _cube(jobs[0][0], seed, DTYPES[case["store"]])
    if kind == "stats":
        n, total, sq = cube.numel(), 0.0, 0.0
        for s in cube:
            total += s.double().sum().item()
        for s in cube:
            sq += ((s.double() - total / n) ** 2).sum().item()
        return dict(moments=dict(count=None, mean=total / n, sd=math.sqrt(sq / n), min=cube.min().item(),
                                 max=cube.max().item()), histogram=None,
                    median=cube.reshape(-1).kthvalue((n + 1) // 2).values.item() if n < 1 << 30 else None)
    field, views = _Field(cube, tf, lo, hi), [_View(d, cam, step) for d, cam in jobs]
    if kind == "sigma":
        mm = _regions(cube, case["region"])
        view = views[0]
        c, t, _ = _render64(view, field, ert, _sigma_units(view, field, mm, case["region"]))
        return dict(minimap=mm, image=_image(c, t, view), nsamples=None)
    if kind == "mip":
        view = views[0]
        m = torch.full(view.n.shape, -math.inf, dtype=torch.float64, device="cuda")

        def visit(rays, k, cell, v):
            m[rays] = torch.maximum(m[rays], v)

        _march(view, field, visit)
        e = field.look_up(m)[2] * (view.n > 0)[:, None]
        return _image(e[:, :3] * e[:, 3:], 1.0 - e[:, 3], view), None
    if kind == "view":
        return _image(*_render64(views[0], field, ert)[:2], views[0]), None
    if kind == "sortlast":
        return dict(image=_image(*_render64(views[0], field, ert)[:2], views[0]), parts=None)
    gtf = torch.zeros((K, 4), dtype=torch.float64, device="cuda")
    gvox = torch.zeros(cube.numel(), dtype=torch.float64, device="cuda")
    images, loss = [], None
    for q, view in enumerate(views):
        c, t, used = _render64(view, field, ert)
        goal = _goal(case, jobs[q][1], seed + q).double()
        off = _image(c, t, view) - goal
        loss = (off ** 2).mean()
        _adjoint64(view, field, c, t, used, 2.0 / goal.numel() * off, gtf, gvox)
        images.append((_image(c, t, view), None))
    gvox = gvox.reshape(cube.shape)
    if kind == "fit":
        return dict(images=images, table=gtf, voxels=gvox)
    return dict(loss=loss, image=images[0][0], table=gtf, voxels=gvox)

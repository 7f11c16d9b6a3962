"""Timed cases: the calls that users of this package make, over the sizes they make them at.

A case names an operation ("op"), a printer and the storage types.  The operations are the
projection operator (volume -> projections), the dose operator (projections -> dose), the
projection optimiser, one differentiable step (dose, thresholded loss, its gradient with
respect to the projections), the voxel error rate, and one convolution layer of the
warm-start network in both directions.

Printers are those of the package's workloads (full grids and pixel arrays; the larger ones
with fewer, still evenly spaced, angles, which scales a pass but not its shape) and, in
draw(), printers of the same kind with other extents, odd ones among them.  Targets are
seeded unions of spheres and boxes inside the region the rays reach; the dose's inputs are
such parts' shadows (line integrals through spheres), a third to a half of them nonzero, as the
optimiser's clamped projections are.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_03516_gb300 import autograd as AG
from paper_2211_03516_gb300 import inputs as I
from paper_2211_03516_gb300 import unet as U
from paper_2211_03516_gb300 import vamrt as V

DEV = "cuda:0"
DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}

# printers of the package's workloads, as plain values
TINY = dict(nx=64, ny=64, nz=64, h=0.2, nu=64, nv=64, angles=90, pupil_mm=150.0, fnum=0.0, pattern="chief", rays=1,
            r_in=6.0, wall=1.0, mu=0.05)
WARM = dict(nx=128, ny=128, nz=128, h=0.1, nu=128, nv=128, angles=180, pupil_mm=100.0, fnum=4.0, pattern="sunflower",
            rays=4, r_in=6.0, wall=1.0, mu=0.05)
MID = dict(nx=256, ny=256, nz=256, h=0.1, nu=256, nv=256, angles=120, pupil_mm=120.0, fnum=4.0,
           pattern="stratified4x4", rays=16, r_in=12.5, wall=1.2, mu=0.03)
TALL = dict(nx=384, ny=384, nz=512, h=0.08, nu=384, nv=512, angles=48, pupil_mm=80.0, fnum=4.0, pattern="sunflower",
            rays=8, r_in=15.0, wall=1.2, mu=0.03)
LARGE = dict(nx=768, ny=768, nz=1024, h=0.05, nu=1024, nv=1024, angles=16, pupil_mm=100.0, fnum=2.8,
             pattern="sunflower", rays=4, r_in=19.0, wall=1.5, mu=0.02)


def listed():
    return [
        # the smallest projection: 64^3, chief rays; launches and per-ray set-up count
        dict(name="project_tiny", op="project", vol="f32", proj="f32", **TINY),
        # the whole method on the smallest printer: five optimiser iterations with their
        # stop checks, as an interactive user runs them
        dict(name="optimise_tiny", op="optimise", iters=5, **TINY),
        # odd extents, an odd number of angles, 13 rays per pixel: nothing divides anything
        dict(name="dose_ragged", op="dose", proj="f32", dose="f32", nx=71, ny=67, nz=53, h=0.19, nu=61, nv=47,
             angles=45, pupil_mm=60.0, fnum=3.5, pattern="hex13", rays=13, r_in=6.2, wall=0.9, mu=0.05),
        # the 256^3 workload: 16 rays per pixel, jittered per pixel, so neighbouring rays
        # spread over several voxels
        dict(name="project_mid", op="project", vol="f32", proj="f32", **MID),
        dict(name="dose_mid", op="dose", proj="f32", dose="f32", **MID),
        # the tall build with BF16 storage: the gradient's projection (signed volume, FP32
        # result) and the dose of BF16 projections
        dict(name="project_tall_bf16", op="project", vol="bf16", proj="f32", **TALL),
        dict(name="dose_tall_bf16", op="dose", proj="bf16", dose="bf16", **TALL),
        # the large print: a 2.4 GB volume and a megapixel array, the headline workload's
        # two operators
        dict(name="project_large", op="project", vol="f32", proj="f32", **LARGE),
        dict(name="dose_large", op="dose", proj="f32", dose="f32", **LARGE),
        # one step of a user's own optimiser through torch.autograd on the 128^3 workload
        dict(name="gradient_warm", op="gradient", **WARM),
        # the quality of a finished dose, the stop check of every loop written outside the
        # library
        dict(name="ver_tall", op="ver", dose="bf16", **{**TALL, "angles": 1}),
        # the widest layer of the warm-start network at the workload's size, forward,
        # weight gradient and data gradient
        dict(name="conv_dec0a", op="conv", d=184, h=128, w=128, cin=48, cout=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: no drawn printer case has more samples than the largest listed one
MOST_SAMPLES = 5.0e10


def draw(rng):
    op = rng.choice(["project", "project", "project", "dose", "dose", "dose", "optimise", "gradient", "ver", "conv"])
    if op == "conv":
        # layers of the network's channel counts over its levels' extents
        cin, cout = rng.choice([(16, 16), (16, 32), (32, 32), (48, 16), (96, 32), (64, 64), (32, 64), (192, 64)])
        w = _log(rng, 16, 128) // 16 * 16      # the weight gradient takes multiples of 16
        d, h = _log(rng, 8, 184), _log(rng, 12, 128)
        while d * h * w * cin * cout > 184 * 128 * 128 * 48 * 16:
            d, h = max(8, d // 2), max(12, h * 3 // 4)
        return dict(op="conv", d=d, h=h, w=w, cin=cin, cout=cout)
    nx = _log(rng, 40, 400)
    ny = nx if rng.random() < 0.7 else nx + rng.randrange(1, 12)
    nz = _log(rng, 24, 500)
    h = rng.choice([0.05, 0.08, 0.1, 0.2])
    rays, pattern = rng.choice([(1, "chief"), (4, "sunflower"), (8, "sunflower"), (13, "hex13"), (16, "stratified4x4")])
    # scans are mostly whole fractions of a degree grid (the workloads' 90, 180, 360 ...);
    # any other count is as legal
    angles = rng.choice([12, 24, 36, 45, 60, 72, 90, 120, 180, 360]) if rng.random() < 0.7 else rng.randrange(5, 200)
    c = dict(op=op, nx=nx, ny=ny, nz=nz, h=h, nu=max(16, int(nx * rng.uniform(0.85, 1.3))),
             nv=max(16, int(nz * rng.uniform(0.85, 1.1))), angles=angles,
             pupil_mm=round(rng.uniform(4.0, 12.0) * nx * h, 3), fnum=0.0 if rays == 1 else rng.choice([2.8, 3.5, 4.0]),
             pattern=pattern, rays=rays, r_in=round(nx * h * rng.uniform(0.44, 0.495), 4),
             wall=round(nx * h * 0.06, 4), mu=rng.choice([0.02, 0.03, 0.05]))
    most = MOST_SAMPLES / {"optimise": 6.0, "gradient": 2.0}.get(op, 1.0)
    while _samples(c) > most and c["angles"] > 4:
        c["angles"] = max(4, c["angles"] // 2)
    if op == "project":
        c.update(vol=rng.choice(["f32", "f32", "bf16", "f16"]), proj=rng.choice(["f32", "f32", "bf16"]))
    elif op == "dose":
        c.update(proj=rng.choice(["f32", "f32", "bf16"]), dose=rng.choice(["f32", "f32", "bf16"]))
    elif op == "optimise":
        c.update(iters=rng.randrange(1, 4))
    elif op == "ver":
        c.update(dose=rng.choice(["f32", "bf16"]), angles=1)
    return c


# ---- inputs ---------------------------------------------------------------------------
def _workload(c):
    fnum = c["fnum"] if c["fnum"] > 0 else I.INF
    return I.Workload(name="case", nx=c["nx"], ny=c["ny"], nz=c["nz"], voxel_mm=c["h"], nu=c["nu"], nv=c["nv"],
                      pixel_u_mm=c["h"], pixel_v_mm=c["h"], n_angles=c["angles"], pupil_mm=c["pupil_mm"],
                      f_number=fnum, pupil_pattern=c["pattern"], rays_per_pixel=c["rays"], r_inner_mm=c["r_in"],
                      wall_mm=c["wall"], n_outside=1.0, n_glass=1.47, n_resin=1.50, mu_per_mm=c["mu"])


def _pupil(c):
    """The printer's aperture: the workloads' own patterns; the sunflower as an explicit list
    of stop points, as a user with a measured aperture passes it."""
    if c["pattern"] == "sunflower":
        return _stop_points(c)
    return I.workload_pupil(_workload(c))


def _stop_points(c):
    m = c["rays"]
    if c["pattern"] == "chief":
        return np.zeros((1, 2))
    if c["pattern"] == "hex13":
        k = np.arange(6)
        a = np.stack([np.cos(k * np.pi / 3), np.sin(k * np.pi / 3)], 1)
        b = np.stack([np.cos(np.pi / 6 + k * np.pi / 3), np.sin(np.pi / 6 + k * np.pi / 3)], 1)
        return np.concatenate([np.zeros((1, 2)), 0.5 * a, 0.5 * math.sqrt(3.0) * b])
    if c["pattern"] == "sunflower":
        k = np.arange(m)
        r, t = np.sqrt((k + 0.5) / m), k * np.pi * (3.0 - math.sqrt(5.0))
        return np.stack([r * np.cos(t), r * np.sin(t)], 1)
    return None


def _reach(c):
    """Radius (mm) that rays reach from every direction, as the workloads' targets use it."""
    return max(min(c["nu"] * c["h"] / 2, c["r_in"] + c["wall"], 1.47 * c["r_in"]) / 1.50 - 1.5 * c["h"], 2 * c["h"])


def _primitives(c, rng, n=14):
    """(centre, radius or half extents) of seeded spheres and boxes inside the reach."""
    reach, zmax = _reach(c), c["nz"] * c["h"] / 2
    scale = min(reach, zmax)
    got = []
    for k in range(n):
        r = rng.uniform(0.12, 0.32) * scale
        rad, phi = (reach - r) * math.sqrt(rng.random()), 2 * math.pi * rng.random()
        z = rng.uniform(-1.0, 1.0) * max(zmax - r - c["h"], 0.0)
        got.append(((rad * math.cos(phi), rad * math.sin(phi), z), r, k % 3 == 2))
    return got


def _part(c, seed):
    """Binary part [nz][ny][nx], FP32."""
    rng = np.random.default_rng(seed)

    def axis(n):
        return (torch.arange(n, device=DEV, dtype=torch.float32) - (n - 1) / 2.0) * c["h"]

    X, Y, Z = axis(c["nx"])[None, None, :], axis(c["ny"])[None, :, None], axis(c["nz"])[:, None, None]
    m = torch.zeros((c["nz"], c["ny"], c["nx"]), device=DEV, dtype=torch.bool)
    for (x, y, z), r, box in _primitives(c, rng):
        lo = max(0, int((z - r) / c["h"] + (c["nz"] - 1) / 2.0))
        hi = min(c["nz"], int((z + r) / c["h"] + (c["nz"] - 1) / 2.0) + 2)
        Zs = Z[lo:hi]
        if box:
            q = 0.7 * r
            m[lo:hi] |= ((X - x).abs() <= q) & ((Y - y).abs() <= q) & ((Zs - z).abs() <= q)
        else:
            m[lo:hi] |= (X - x) ** 2 + (Y - y) ** 2 + (Zs - z) ** 2 <= r * r
    return m.float()


def _shadows(c, seed):
    """Projections [angles][nv][nu] of seeded spheres: chord lengths where the printer's
    rays cross them (the vial magnifies u by about the resin's index)."""
    rng = np.random.default_rng(seed)
    u = (torch.arange(c["nu"], device=DEV, dtype=torch.float32) - (c["nu"] - 1) / 2.0) * c["h"]
    v = (torch.arange(c["nv"], device=DEV, dtype=torch.float32) - (c["nv"] - 1) / 2.0) * c["h"]
    g = torch.zeros((c["angles"], c["nv"], c["nu"]), device=DEV)
    th = torch.arange(c["angles"], device=DEV, dtype=torch.float32) * (2 * math.pi / c["angles"])
    for (x, y, z), r, _ in _primitives(c, rng, 30):
        uc = 1.5 * (torch.cos(th) * x + torch.sin(th) * y)
        d2 = ((u[None, :] - uc[:, None]) / 1.5) ** 2
        g += 2 * (r * r - d2[:, None, :] - ((v - z) ** 2)[None, :, None]).clamp_min(0).sqrt()
    return g


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if c["op"] == "conv":
        pos = (c["d"], c["h"], c["w"])
        x = torch.randn(pos + (c["cin"],), device=DEV, generator=gen).relu().to(torch.bfloat16)
        dy = (torch.randn(pos + (c["cout"],), device=DEV, generator=gen) * 0.01).to(torch.bfloat16)
        w = (torch.randn((c["cout"], 27, c["cin"]), device=DEV, generator=gen) * (2.0 / (27 * c["cin"])) ** 0.5)
        b = torch.randn(c["cout"], device=DEV, generator=gen) * 0.1
        w = w.to(torch.bfloat16)
        # the data gradient's weights: taps reversed, channels swapped
        wt = w.flip(1).permute(2, 1, 0).contiguous()
        return dict(case=c, x=x, dy=dy, w=w, b=b, wt=wt)
    s = dict(case=c, P=V.Projector.from_workload(_workload(c), _pupil(c)))
    if c["op"] == "project":
        f = _part(c, seed)
        if c["vol"] == "f32":       # a model: the part, its values spread by the updates
            f.mul_(torch.rand(f.shape, device=DEV, generator=gen).add_(0.5))
        else:                       # a loss gradient: negative in the part, positive around it
            f = torch.rand(f.shape, device=DEV, generator=gen) * (0.3 - f)
        s["vol"] = f.to(DT[c["vol"]])
    elif c["op"] == "dose":
        s["proj"] = _shadows(c, seed).to(DT[c["proj"]])
    elif c["op"] == "optimise":
        s["target"] = _part(c, seed)
    elif c["op"] == "gradient":
        s["target"] = _part(c, seed)
        s["proj"] = _shadows(c, seed) / (c["angles"] * _reach(c))
    elif c["op"] == "ver":
        s["target"] = _part(c, seed)
        d = torch.rand(s["target"].shape, device=DEV, generator=gen) * 0.5 + 0.4 * s["target"]
        s["dose"] = d.to(DT[c["dose"]])
    return s


def run(state):
    c, op = state["case"], state["case"]["op"]
    if op == "project":
        return state["P"].adjoint(state["vol"], proj_dtype=DT[c["proj"]])
    if op == "dose":
        return state["P"].forward_dose(state["proj"], dose_dtype=DT[c["dose"]])
    if op == "optimise":
        res = state["P"].optimize(state["target"], max_iter=c["iters"], tol=0.0)
        return dict(proj=res["proj"], dose=res["dose"], model=res["model"])
    if op == "gradient":
        g = state["proj"].detach().requires_grad_(True)
        d = AG.dose(g, state["P"])
        loss = AG.threshold_loss(d, state["target"], state["P"], 0.8, 1.0)
        loss.backward()
        return dict(loss=loss.detach().float(), dose=d.detach(), grad=g.grad)
    if op == "ver":
        ver, index = state["P"].voxel_error_rate(state["dose"], state["target"])
        return dict(ver=ver, index=index)
    y = U.conv3d(state["x"], state["w"], state["b"], relu=True)
    dw = torch.zeros((c["cout"], 27, c["cin"]), device=DEV)
    U.conv3d_wgrad(state["x"], state["dy"], dw, 27)
    dx = U.conv3d(state["dy"], state["wt"])
    return dict(y=y, dw=dw, dx=dx)


# ---- what a pass cannot do without ------------------------------------------------------
def _samples(c):
    """Samples of a pass (two per voxel of path in the resin), over all rays."""
    u = (np.arange(c["nu"]) - (c["nu"] - 1) / 2.0) * c["h"] / 1.50
    chord = 2 * np.sqrt(np.maximum(c["r_in"] ** 2 - u ** 2, 0.0))
    return float(chord.sum() * 2 / c["h"] * c["nv"] * c["rays"] * c["angles"])


def work(case):
    c = case
    size = {"f32": 4, "bf16": 2, "f16": 2}
    if c["op"] == "conv":
        n = c["d"] * c["h"] * c["w"]
        return dict(bytes=2.0 * n * (2 * c["cin"] + 2 * c["cout"]) + 3 * 4.0 * 27 * c["cin"] * c["cout"],
                    flops=3 * 2.0 * n * 27 * c["cin"] * c["cout"])
    vox, pix = float(c["nx"] * c["ny"] * c["nz"]), float(c["angles"] * c["nv"] * c["nu"])
    # a sample: eight weights (12 operations with its attenuation) and eight multiply-adds
    per = 28.0 * _samples(c)
    if c["op"] == "project":
        return dict(bytes=vox * size[c["vol"]] + pix * size[c["proj"]], flops=per)
    if c["op"] == "dose":
        return dict(bytes=vox * size[c["dose"]] + pix * size[c["proj"]], flops=per)
    if c["op"] == "optimise":
        return dict(bytes=c["iters"] * (2 * pix * 4 + 5 * vox * 4), flops=c["iters"] * 2 * per)
    if c["op"] == "gradient":
        return dict(bytes=2 * pix * 4 + 2 * vox * 4, flops=2 * per)
    return dict(bytes=vox * (size[c["dose"]] + 4), flops=4 * vox)


# ---- the same in 64 bits ---------------------------------------------------------------
class _Exact:
    """The printer's dose matrix applied sample by sample in FP64 (torch)."""

    def __init__(self, c):
        self.c = c
        f8 = dict(device=DEV, dtype=torch.float64)
        h, R, Ro = c["h"], c["r_in"], c["r_in"] + c["wall"]
        xy = torch.from_numpy(np.ascontiguousarray(_stop_points(c))).to(**f8)
        M, nu, nv = c["rays"], c["nu"], c["nv"]
        u = (torch.arange(nu, **f8) - (nu - 1) / 2.0) * h
        v = (torch.arange(nv, **f8) - (nv - 1) / 2.0) * h
        Q = torch.stack([u[None, None, :].expand(M, nv, nu), torch.zeros((M, nv, nu), **f8),
                         v[None, :, None].expand(M, nv, nu)], -1)
        D = c["pupil_mm"] / c["fnum"] if c["fnum"] > 0 else 0.0
        o = torch.stack([0.5 * D * xy[:, 0], torch.full((M,), -c["pupil_mm"], **f8), 0.5 * D * xy[:, 1]], -1)
        o = o[:, None, None, :].expand_as(Q)
        d = Q - o
        d = d / d.norm(dim=-1, keepdim=True)
        ok = torch.ones((M, nv, nu), device=DEV, dtype=torch.bool)

        def enter(p, d, r):      # first crossing of the cylinder of radius r
            a = d[..., 0] ** 2 + d[..., 1] ** 2
            b = p[..., 0] * d[..., 0] + p[..., 1] * d[..., 1]
            disc = b * b - a * (p[..., 0] ** 2 + p[..., 1] ** 2 - r * r)
            t = (-b - disc.clamp_min(0).sqrt()) / a
            return p + t[..., None] * d, (disc >= 0) & (t > 0)

        def bend(p, d, r, n1, n2):
            n = torch.cat([p[..., :2] / r, torch.zeros_like(p[..., :1])], -1)     # outward, against d
            ci = -(n * d).sum(-1)
            k = 1 - (n1 / n2) ** 2 * (1 - ci * ci)
            ct = k.clamp_min(0).sqrt()
            out = (n1 / n2) * d + ((n1 / n2) * ci - ct)[..., None] * n
            rs = (n1 * ci - n2 * ct) / (n1 * ci + n2 * ct)
            rp = (n1 * ct - n2 * ci) / (n1 * ct + n2 * ci)
            return out, 1 - (rs * rs + rp * rp) / 2, k >= 0

        p, hit = enter(o, d, Ro)
        ok &= hit
        d, T1, hit = bend(p, d, Ro, 1.0, 1.47)
        ok &= hit
        e, hit = enter(p, d, R)
        ok &= hit
        d, T2, hit = bend(e, d, R, 1.47, 1.50)
        ok &= hit
        ell = -2 * (e[..., 0] * d[..., 0] + e[..., 1] * d[..., 1]) / (d[..., 0] ** 2 + d[..., 1] ** 2)
        ok &= ell > 0
        K = torch.ceil(torch.where(ok, ell, 0.0) / (0.5 * h) - 1e-9).clamp_min(1)
        delta = ell / K
        self.K = torch.where(ok, K, 0.0).long()
        self.most = int(self.K.max())
        j = torch.arange(self.most, **f8) + 0.5
        self.s = delta[..., None] * j                                    # mm along the ray
        live = ok[..., None] & (torch.arange(self.most, device=DEV) < self.K[..., None])
        w = (T1 * T2 * delta / M)[..., None] * torch.exp(-c["mu"] * self.s)
        self.w = torch.where(live, w, 0.0)
        self.e, self.d = torch.where(ok[..., None], e, 0.0), torch.where(ok[..., None], d, 0.0)
        self.s = torch.where(live, self.s, 0.0)
        self.th = 2 * math.pi * np.arange(c["angles"]) / c["angles"]

    def _cells(self, k):
        """Per sample: flat index of its lower corner in the grid with two halo voxels, and
        the three fractions."""
        c, (cs, sn) = self.c, (math.cos(self.th[k]), math.sin(self.th[k]))
        pos = [(cs * self.e[..., 0] - sn * self.e[..., 1], cs * self.d[..., 0] - sn * self.d[..., 1], c["nx"]),
               (sn * self.e[..., 0] + cs * self.e[..., 1], sn * self.d[..., 0] + cs * self.d[..., 1], c["ny"]),
               (self.e[..., 2], self.d[..., 2], c["nz"])]
        idx, frac = [], []
        for a, b, n in pos:
            q = (a[..., None] + b[..., None] * self.s) / c["h"] + (n - 1) / 2.0
            i = q.floor()
            frac.append(q - i)
            idx.append((i.long() + 2).clamp_(0, n + 2))
        return (idx[2] * (c["ny"] + 4) + idx[1]) * (c["nx"] + 4) + idx[0], frac

    def _corners(self, k):
        c = self.c
        base, (fx, fy, fz) = self._cells(k)
        sx, sxy = c["nx"] + 4, (c["nx"] + 4) * (c["ny"] + 4)
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    wt = (fx if dx else 1 - fx) * (fy if dy else 1 - fy) * (fz if dz else 1 - fz)
                    yield base + (dz * sxy + dy * sx + dx), wt

    def project(self, vol):
        v = torch.nn.functional.pad(vol.double(), (2, 2, 2, 2, 2, 2)).reshape(-1)
        out = []
        for k in range(len(self.th)):
            acc = torch.zeros_like(self.w)
            for idx, wt in self._corners(k):
                acc += wt * v[idx]
            out.append((acc * self.w).sum(-1).sum(0))
        return torch.stack(out)

    def dose(self, proj):
        c = self.c
        v = torch.zeros((c["nz"] + 4) * (c["ny"] + 4) * (c["nx"] + 4), device=DEV, dtype=torch.float64)
        for k in range(len(self.th)):
            g = proj[k].double()[None, :, :, None] * self.w
            for idx, wt in self._corners(k):
                v.scatter_add_(0, idx.reshape(-1), (wt * g).reshape(-1))
        return v.view(c["nz"] + 4, c["ny"] + 4, c["nx"] + 4)[2:-2, 2:-2, 2:-2].contiguous()


def _loss(d, f, lo, hi):
    p, q = (hi - d).clamp_min(0) * (f > 0.5), (d - lo).clamp_min(0) * (f <= 0.5)
    np_, nq = (f > 0.5).sum().clamp_min(1), (f <= 0.5).sum().clamp_min(1)
    return (p * p).sum() / np_ + (q * q).sum() / nq, 2 * (q / nq - p / np_)


def _resin(c):
    x = (torch.arange(c["nx"], device=DEV, dtype=torch.float64) - 0.5 * (c["nx"] - 1)) * c["h"]
    y = (torch.arange(c["ny"], device=DEV, dtype=torch.float64) - 0.5 * (c["ny"] - 1)) * c["h"]
    return (x * x)[None, :] + (y * y)[:, None] <= c["r_in"] * c["r_in"]


def _conv64(x, w):
    """'Same' 3 x 3 x 3 convolution, channels last, taps in (z, y, x) order."""
    D, H, W, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    y = torch.zeros((D, H, W, w.shape[0]), device=x.device, dtype=x.dtype)
    for t in range(27):
        a, b, e = t // 9, t // 3 % 3, t % 3
        y += xp[a:a + D, b:b + H, e:e + W] @ w[:, t].T
    return y


def exact(case, seed):
    c = case
    if c["op"] == "conv":
        s = prepare(c, seed)
        x, dy, D, H, W = s["x"].double(), s["dy"].double(), c["d"], c["h"], c["w"]
        y = (_conv64(x, s["w"].double()) + s["b"].double()).clamp_min(0)
        xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
        g = dy.reshape(-1, c["cout"])
        dw = torch.stack([g.T @ xp[t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W].reshape(-1, c["cin"])
                          for t in range(27)], 1)
        return dict(y=y, dw=dw, dx=_conv64(dy, s["wt"].double()))
    if c["op"] == "ver":
        s = prepare(c, seed)
        # the rate is defined by FP32 bins of the stored dose
        x, f = s["dose"].float()[:, _resin(c)], s["target"][:, _resin(c)]
        b = torch.floor(x * (1024.0 / x.max())).clamp(0, 1023).long()
        below = torch.bincount(b[f > 0.5], minlength=1024).cumsum(0)[:-1]
        above = (f <= 0.5).sum() - torch.bincount(b[f <= 0.5], minlength=1024).cumsum(0)[:-1]
        best = int((below + above).argmin())
        return dict(ver=float(below[best] + above[best]) / x.numel(), index=best + 1)
    work_ = _samples(c) * {"optimise": 2 * c.get("iters", 1), "gradient": 2}.get(c["op"], 1)
    if _stop_points(c) is None or work_ > 6e9 or _samples(c) / c["angles"] > 1.2e8:
        return None
    E = _Exact(c)
    s = prepare(c, seed)
    if c["op"] == "project":
        return E.project(s["vol"])
    if c["op"] == "dose":
        return E.dose(s["proj"])
    if c["op"] == "gradient":
        d = E.dose(s["proj"])
        loss, gd = _loss(d, s["target"].double(), 0.8, 1.0)
        return dict(loss=loss, dose=d, grad=E.project(gd))
    f = s["target"].double()
    m = f.clone()
    for _ in range(c["iters"]):
        g = E.project(m).clamp_min(0)
        d = E.dose(g)
        dn = d / d[:, _resin(c)].max()
        m = (m + f - dn).clamp_min(0)
    return dict(proj=g, dose=dn, model=m)

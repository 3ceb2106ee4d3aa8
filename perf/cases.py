"""Workloads of the shading framework, through its public entry points.

A case is a dict of plain values; ``kind`` names the work a pass does:

* ``step``    an analysis-by-synthesis step: shade, then every requested
              gradient (``api`` "l2": ``Scene.shade`` + ``Scene.backward_l2``;
              "autograd": the differentiable ``shade`` function)
* ``render``  forward shading only
* ``relight`` radiance from the saved log-visibility (lighting or albedo
              changed, the geometry did not)
* ``serve``   a burst of requests to the continuous-batching server
* ``views``   all views of a posed, deforming mesh: chain, shading, gradients
* ``envmap``  SH lighting from an equirectangular map
* ``raster``  vertex radiance to an image, and the gradients back

Inputs are synthetic, drawn on the device from the seed alone, with the
geometry of ``paper_2104_00359_gb300.synthetic``.  ``exact`` restates every
computation in float64 torch.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2104_00359_gb300 import Config, Scene, _lib, serve, shade, synthetic
from paper_2104_00359_gb300.chain import ViewBatch, render_views_batched
from paper_2104_00359_gb300.envmap import project_envmap
from paper_2104_00359_gb300.raster import rasterize

DEV = "cuda"
EPSILON = 3.0
PRECISION = {"fp32": _lib.SHS_FP32, "bf16": _lib.SHS_BF16, "tf32": _lib.SHS_TF32, "fp16": _lib.SHS_FP16}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The smallest optimisation step: a 32 x 32 plane under 8 spheres, all
        # scene parameters updated through autograd.  Launches and latency.
        dict(name="plane32_step", kind="step", api="autograd", scene="plane", points=1024, spheres=8, bands=4,
             precision="fp32", exp_mode=0, fixed_k=-1, cull=False),
        # The headline step: a 512 x 512 G-buffer of a capsule body with 100
        # occluder spheres, L2 loss, gradients to light, albedo and spheres.
        dict(name="capsule512_step", kind="step", api="l2", scene="capsule", points=512 * 512, spheres=100, bands=4,
             precision="fp32", exp_mode=0, fixed_k=-1, cull=False),
        # A small ragged preview render with horizon culling.
        dict(name="ragged_render", kind="render", scene="field", points=10007, spheres=33, bands=4,
             precision="fp32", exp_mode=0, fixed_k=-1, cull=True),
        # The 8-band megapixel optimisation step (the largest scene).  A fixed
        # number of squarings keeps the loss continuous between steps.
        dict(name="field1024_step_b8", kind="step", api="l2", scene="field", points=1024 * 1024, spheres=300, bands=8,
             precision="fp32", exp_mode=0, fixed_k=5, cull=False),
        # A megapixel 8-band still with the projected exponential (the most
        # accurate variant), forward only.
        dict(name="field1024_render_b8_projexp", kind="render", scene="field", points=1024 * 1024, spheres=300,
             bands=8, precision="fp32", exp_mode=1, fixed_k=-1, cull=False),
        # The same optimisation at 512 x 512 on the tensor cores.
        dict(name="field512_step_b8_bf16", kind="step", api="l2", scene="field", points=512 * 512, spheres=300,
             bands=8, precision="bf16", exp_mode=0, fixed_k=5, cull=False),
        # Texture / lighting optimisation over fixed geometry: the forward
        # from saved pair terms, a ragged 6-band job.
        dict(name="relight_b6", kind="relight", scene="field", points=200003, spheres=150, bands=6,
             precision="fp32", exp_mode=0, fixed_k=-1, cull=False),
        # Eight resident jobs of the serving mix (4 and 6 bands), one burst of
        # requests, two in three with the loss and its gradients.
        dict(name="serve_mix8", kind="serve", jobs=8, min_points=16384, max_points=131072, min_spheres=20,
             max_spheres=300),
        # Multi-view mesh optimisation: 16 posed views of a 50,000-vertex
        # mesh, 200 spheres, 60 deformation parameters.
        dict(name="mesh16_views_step", kind="views", views=16, theta=250, phi=200, spheres=200, params=60, bands=4,
             fixed_k=4),
        # Lighting set-up from a full-size HDR panorama.
        dict(name="envmap_4096x8192_b8", kind="envmap", height=4096, width=8192, bands=8),
        # Lighting from a small panorama of odd size.
        dict(name="envmap_500x1001_b4", kind="envmap", height=500, width=1001, bands=4),
        # Image-space loss on the mesh: 50,000 shaded vertices to a megapixel
        # image and the image gradient back to radiance and positions.
        dict(name="raster1024_step", kind="raster", theta=250, phi=200, height=1024, width=1024),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "render", "render", "relight", "serve", "views", "envmap", "raster"])
    if kind in ("step", "render", "relight"):
        bands = rng.choice([3, 4, 4, 5, 6, 8, 8])
        spheres = _log_int(rng, 8, 300)
        top = 1000000 if bands <= 4 else 400000
        c = dict(kind=kind, scene=rng.choice(["field", "plane"]), points=_log_int(rng, 1000, top), spheres=spheres,
                 bands=bands, precision="fp32", exp_mode=0, fixed_k=-1, cull=rng.random() < 0.25)
        if kind == "step":
            c["api"] = rng.choice(["l2", "autograd"])
            if bands == 8 and rng.random() < 0.4:
                c["precision"] = rng.choice(["bf16", "tf32", "fp16"])
            # large optimisations fix the squaring count (a continuous loss)
            c["fixed_k"] = 5 if c["points"] > 30000 else -1
        else:
            c["exp_mode"] = 1 if bands >= 5 else rng.choice([0, 0, 1])
        return c
    if kind == "serve":
        hi = _log_int(rng, 20000, 131072)
        return dict(kind=kind, jobs=rng.randint(2, 10), min_points=rng.randint(2000, 16384), max_points=hi,
                    min_spheres=20, max_spheres=rng.randint(60, 300))
    if kind == "views":
        return dict(kind=kind, views=rng.randint(2, 20), theta=rng.randint(20, 250), phi=rng.randint(24, 200),
                    spheres=_log_int(rng, 20, 300), params=rng.randint(6, 130), bands=rng.choice([3, 4]), fixed_k=4)
    if kind == "envmap":
        h = _log_int(rng, 64, 4096)
        w = rng.choice([2 * h, 2 * h + 1, 16 * (h // 8)])
        return dict(kind=kind, height=h, width=w, bands=rng.choice([3, 4, 5, 6, 8]))
    return dict(kind=kind, theta=rng.randint(20, 300), phi=rng.randint(24, 300), height=_log_int(rng, 100, 1500),
                width=_log_int(rng, 100, 1500))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Draw:
    """Float64 random numbers on the device from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) & 0x7FFFFFFF)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def normal(self, sigma, *shape):
        return sigma * torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64)


def _f32(t):
    return t.to(torch.float32).contiguous()


def _lighting(rng, bands, decay):
    K = bands * bands
    L = rng.normal(0.3, 3, K)
    if decay:
        L = L / (torch.arange(K, device=DEV, dtype=torch.float64).sqrt().floor() + 1.0)
    L[:, 0] = 1.0
    return L


def _grid(points):
    res = math.isqrt(points - 1) + 1
    t = -1.0 + (2.0 * torch.arange(res, device=DEV, dtype=torch.float64) + 1.0) / res
    y, x = torch.meshgrid(t, t, indexing="ij")
    return x.reshape(-1)[:points], y.reshape(-1)[:points]


def _plane(rng, points, spheres, bands):
    x, y = _grid(points)
    z = torch.zeros_like(x)
    centers = torch.cat([rng.uniform(-0.8, 0.8, spheres, 2), rng.uniform(0.1, 0.6, spheres, 1)], 1)
    return dict(points=torch.stack([x, y, z], 1), normals=torch.stack([z, z, z + 1.0], 1),
                albedo=torch.full((points, 3), 0.5, device=DEV, dtype=torch.float64), centers=centers,
                radii=rng.uniform(0.05, 0.2, spheres), light=_lighting(rng, bands, False))


def _field(rng, points, spheres, bands, bumps=16):
    amp, mu, sig = rng.uniform(-0.25, 0.25, bumps), rng.uniform(-1, 1, bumps, 2), rng.uniform(0.1, 0.4, bumps)

    def height(x, y):
        h, hx, hy = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
        for b in range(bumps):
            dx, dy, s2 = x - mu[b, 0], y - mu[b, 1], sig[b] ** 2
            g = amp[b] * torch.exp(-(dx * dx + dy * dy) / (2 * s2))
            h, hx, hy = h + g, hx - g * dx / s2, hy - g * dy / s2
        return h, hx, hy

    x, y = _grid(points)
    h, hx, hy = height(x, y)
    n = torch.stack([-hx, -hy, torch.ones_like(h)], 1)
    c = rng.uniform(-1, 1, spheres, 2)
    cz = height(c[:, 0], c[:, 1])[0] + rng.uniform(0.05, 0.8, spheres)
    radii = torch.exp(rng.uniform(math.log(0.01), math.log(0.2), spheres))
    return dict(points=torch.stack([x, y, h], 1), normals=n / n.norm(dim=1, keepdim=True),
                albedo=rng.uniform(0.2, 0.9, points, 3), centers=torch.cat([c, cz[:, None]], 1), radii=radii,
                light=_lighting(rng, bands, True))


def _capsule(rng, points, spheres, bands, per_bone=5, along=24):
    """Top-down G-buffer of a random-walk chain of capsules above a plane."""
    bones = spheres // per_bone
    lo = torch.tensor([-0.85, -0.85, 0.28], dtype=torch.float64)
    hi = torch.tensor([0.85, 0.85, 1.6], dtype=torch.float64)
    start, steps = rng.uniform(0.3, 0.7, 3).cpu(), rng.normal(1.0, bones, 3).cpu()
    length = rng.uniform(0.12, 0.22, bones).cpu()
    joints = [lo + (hi - lo) * start]
    for b in range(bones):
        nxt = joints[-1] + steps[b] / steps[b].norm() * length[b]
        nxt = torch.where(nxt < lo, 2 * lo - nxt, nxt)
        joints.append(torch.where(nxt > hi, 2 * hi - nxt, nxt))
    joints = torch.stack(joints).to(DEV)
    a, e = joints[:-1], joints[1:]
    ts = (torch.arange(per_bone, device=DEV, dtype=torch.float64) + 0.5) / per_bone
    centers = (a[:, None] + ts[None, :, None] * (e - a)[:, None]).reshape(-1, 3)
    radii = rng.uniform(0.02, 0.12, bones, per_bone)
    x, y = _grid(points)
    z = torch.zeros_like(x)
    n = torch.stack([z, z, z + 1.0], 1)
    us = torch.linspace(0, 1, along, device=DEV, dtype=torch.float64)
    for b in range(bones):
        R = radii[b].max() + 0.01
        c = a[b] + us[:, None] * (e[b] - a[b])
        h2 = R * R - (x[None] - c[:, :1]) ** 2 - (y[None] - c[:, 1:2]) ** 2
        hit = torch.where(h2 > 0, c[:, 2:] + h2.clamp(min=0).sqrt(), torch.full_like(h2, -1.0))
        top, at = hit.max(0)
        better = top > z
        z = torch.where(better, top, z)
        m = (torch.stack([x, y, top], 1) - c[at]) / R
        n = torch.where(better[:, None], m, n)
    return dict(points=torch.stack([x, y, z], 1), normals=n / n.norm(dim=1, keepdim=True),
                albedo=rng.uniform(0.2, 0.9, points, 3), centers=centers, radii=radii.reshape(-1),
                light=_lighting(rng, bands, False))


def _scene(case, seed):
    make = {"plane": _plane, "field": _field, "capsule": _capsule}[case["scene"]]
    rng = _Draw(seed)
    s = {k: _f32(v) for k, v in make(rng, case["points"], case["spheres"], case["bands"]).items()}
    s["target"] = _f32(rng.uniform(0.0, 0.6, case["points"], 3))
    s["d_radiance"] = _f32(rng.normal(1.0, case["points"], 3))
    return s


def _config(case):
    return Config(n_bands=case["bands"], precision=PRECISION[case.get("precision", "fp32")],
                  fixed_k=case.get("fixed_k", -1), horizon_cull=case.get("cull", False),
                  exp_mode=case.get("exp_mode", 0))


def _rank_points(case, j):
    lo, hi = sorted((case["min_points"], case["max_points"]))
    return lo * (hi / lo) ** ((j + 0.5) / case["jobs"])


def _rank_spheres(case, j):
    at = ((5 * j + 2) % case["jobs"] + 0.5) / case["jobs"]
    return case["min_spheres"] + (case["max_spheres"] - case["min_spheres"]) * at


def _serve_jobs(case, seed):
    """Inputs of the jobs of a serving burst, sizes log-uniform over the range."""
    jobs = []
    for j in range(case["jobs"]):
        points, spheres = int(round(_rank_points(case, j))), int(round(_rank_spheres(case, j)))
        bands = 4 if j % 2 else 6
        s = {k: _f32(v) for k, v in _field(_Draw(seed * 64 + j), points, spheres, bands, bumps=4).items()}
        s["target"] = _f32(_Draw(seed * 64 + j + 7919).uniform(0.0, 0.6, points, 3))
        jobs.append(dict(bands=bands, op="fwd" if j % 3 == 2 else "fwdbwd", **s))
    return jobs


def _mesh(case, seed):
    rng = _Draw(seed)
    th = (torch.arange(case["theta"], device=DEV, dtype=torch.float64) + 0.5) / case["theta"] * math.pi
    ph = torch.arange(case["phi"], device=DEV, dtype=torch.float64) / case["phi"] * 2 * math.pi
    t, p = (v.reshape(-1) for v in torch.meshgrid(th, ph, indexing="ij"))
    coef = rng.normal(0.03, 4, 4)
    r, rt, rp = torch.ones_like(t), torch.zeros_like(t), torch.zeros_like(t)
    for a in range(4):
        for b in range(4):
            c = coef[a, b]
            r = r + c * torch.cos((a + 1) * t) * torch.cos(b * p)
            rt = rt - c * (a + 1) * torch.sin((a + 1) * t) * torch.cos(b * p)
            rp = rp - c * b * torch.cos((a + 1) * t) * torch.sin(b * p)
    st, ct, sp, cp = torch.sin(t), torch.cos(t), torch.sin(p), torch.cos(p)
    u = torch.stack([st * cp, st * sp, ct], 1)
    et = rt[:, None] * u + r[:, None] * torch.stack([ct * cp, ct * sp, -st], 1)
    ep = rp[:, None] * u + r[:, None] * torch.stack([-st * sp, st * cp, torch.zeros_like(t)], 1)
    n = torch.linalg.cross(et, ep)
    n = n / n.norm(dim=1, keepdim=True).clamp(min=1e-9)
    n = n * torch.sign((n * u).sum(1, keepdim=True))
    return rng, r[:, None] * u, n


def _views_inputs(case, seed):
    rng, v0, n0 = _mesh(case, seed)
    M, N, D, V = v0.shape[0], case["spheres"], case["params"], case["views"]
    d, w = rng.normal(1.0, N, 3), rng.normal(1.0, V, 3)
    poses = torch.cat([w / w.norm(dim=1, keepdim=True) * rng.uniform(0.0, math.pi, V, 1), rng.normal(0.1, V, 3)], 1)
    s = dict(v0=v0, n0=n0, A_v=rng.normal(0.01, M, 3, D), A_n=rng.normal(0.01, M, 3, D),
             c0=d / d.norm(dim=1, keepdim=True) * rng.uniform(0.4, 0.7, N, 1), A_c=rng.normal(0.01, N, 3, D),
             radii=rng.uniform(0.04, 0.1, N), light=_lighting(rng, case["bands"], False),
             albedo=rng.uniform(0.2, 0.9, M, 3), poses=poses, p=rng.normal(0.1, D),
             d_radiance=rng.normal(1.0, V, M, 3))
    return {k: _f32(v) for k, v in s.items()}


def _raster_inputs(case, seed):
    rng, v0, _ = _mesh(case, seed)
    eye = rng.normal(1.0, 3).cpu().numpy()
    eye = eye / np.linalg.norm(eye) * 3.0
    up = (0.0, 0.0, 1.0) if abs(eye[2]) < 2.5 else (0.0, 1.0, 0.0)
    proj = synthetic.look_at_perspective(eye, up=up, aspect=case["width"] / case["height"])
    t = torch.arange(case["theta"] - 1, device=DEV)[:, None] * case["phi"]
    p = torch.arange(case["phi"], device=DEV)[None]
    a, b = (t + p).reshape(-1), (t + (p + 1) % case["phi"]).reshape(-1)
    faces = torch.stack([torch.stack([a, a + case["phi"], b], 1),
                         torch.stack([b, a + case["phi"], b + case["phi"]], 1)], 1).reshape(-1, 3)
    return dict(vertices=_f32(v0), radiance=_f32(rng.uniform(0.0, 1.0, v0.shape[0], 3)),
                faces=faces.to(torch.int32).contiguous(), proj=proj,
                d_image=_f32(rng.normal(1.0, case["height"], case["width"], 3)))


def _env_inputs(case, seed):
    """A sky gradient over a darker ground, two suns and 5 % noise."""
    rng = _Draw(seed)
    H, W = case["height"], case["width"]
    th = (torch.arange(H, device=DEV, dtype=torch.float32) + 0.5) * (math.pi / H)
    ph = (torch.arange(W, device=DEV, dtype=torch.float32) + 0.5) * (2 * math.pi / W)
    z, s = torch.cos(th)[:, None], torch.sin(th)[:, None]
    zenith, horizon, ground = (_f32(rng.uniform(lo, hi, 3)) for lo, hi in ((0.3, 0.6), (0.7, 1.0), (0.1, 0.3)))
    sky = horizon + (zenith - horizon) * z.clamp(min=0)[..., None]
    env = torch.where(z[..., None] >= 0, sky, ground.expand(H, 1, 3)).expand(H, W, 3).clone()
    for _ in range(2):
        el, az, radius, power = (float(v) for v in torch.stack([
            rng.uniform(0.1, 1.3, 1), rng.uniform(0.0, 6.28, 1), rng.uniform(0.035, 0.087, 1),
            rng.uniform(20.0, 60.0, 1)]).flatten())
        dot = s * math.cos(el) * torch.cos(ph[None] - az) + z * math.sin(el)
        env += ((dot >= math.cos(radius)) * power)[..., None] * _f32(rng.uniform(0.8, 1.0, 3))
    env *= 0.95 + 0.1 * torch.rand(env.shape, generator=rng.g, device=DEV)
    return env


# ---------------------------------------------------------------------------
# preparing and running
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "render", "relight"):
        s = _scene(case, seed)
        s["kind"], s["api"] = kind, case.get("api")
        s["scene"] = Scene(s["centers"], s["radii"], s["light"], _config(case))
        if kind == "step" and s["api"] == "autograd":
            for k in ("albedo", "centers", "radii", "light"):
                s[k].requires_grad_(True)
        elif kind != "render":
            s["saved"] = s["scene"].new_saved(case["points"])
        if kind == "relight":
            s["scene"].shade(s["points"], s["normals"], s["albedo"], saved=s["saved"])
        return s
    if kind == "serve":
        srv, ops = serve.Server(hbm_budget_bytes=20e9), []
        for j, job in enumerate(_serve_jobs(case, seed)):
            srv.add_job(j, job["points"], job["normals"], job["albedo"], job["centers"], job["radii"], job["light"],
                        Config(n_bands=job["bands"]), target=job["target"])
            ops.append(job["op"])
        return dict(kind=kind, server=srv, ops=ops)
    if kind == "views":
        s = _views_inputs(case, seed)
        s["kind"] = kind
        s["views"] = ViewBatch(case["views"], s["v0"].shape[0], s["c0"], s["radii"], s["light"],
                               Config(n_bands=case["bands"], fixed_k=case["fixed_k"]))
        for k in ("p", "poses", "radii", "light", "albedo"):
            s[k].requires_grad_(True)
        return s
    if kind == "envmap":
        return dict(kind=kind, env=_env_inputs(case, seed), bands=case["bands"])
    s = _raster_inputs(case, seed)
    s["vertices"].requires_grad_(True)
    s["radiance"].requires_grad_(True)
    return dict(kind=kind, size=(case["height"], case["width"]), **s)


def run(s):
    kind = s["kind"]
    if kind == "step" and s["api"] == "l2":
        B = s["scene"].shade(s["points"], s["normals"], s["albedo"], saved=s["saved"])
        g = s["scene"].backward_l2(s["points"], s["normals"], s["albedo"], B, s["target"], saved=s["saved"],
                                   want=("light", "albedo", "centers", "radii"))
        return dict(radiance=B, **{k: v for k, v in g.items() if v is not None})
    if kind == "step":
        B = shade(s["points"], s["normals"], s["albedo"], s["centers"], s["radii"], s["light"], s["scene"])
        names = ("albedo", "centers", "radii", "light")
        g = torch.autograd.grad(B, [s[k] for k in names], s["d_radiance"])
        return dict(radiance=B.detach(), **{"d_" + k: v for k, v in zip(names, g)})
    if kind == "render":
        return dict(radiance=s["scene"].shade(s["points"], s["normals"], s["albedo"]))
    if kind == "relight":
        return dict(radiance=s["scene"].shade_tail(s["normals"], s["albedo"], s["saved"]))
    if kind == "serve":
        srv = s["server"]
        for j, op in enumerate(s["ops"]):
            srv.submit(j, op)
        srv.drain()
        srv.completed.clear()
        out = []
        for j, op in enumerate(s["ops"]):
            job = srv.jobs[j]
            grads = dict(job.grads, loss=job.loss) if op == "fwdbwd" else {}
            out.append(dict(radiance=job.radiance, **{k: v for k, v in grads.items() if v is not None}))
        return out
    if kind == "views":
        B = render_views_batched(s["p"], s["poses"], s, s["radii"], s["light"], s["albedo"], s["views"])
        names = ("p", "poses", "radii", "light", "albedo")
        g = torch.autograd.grad(B, [s[k] for k in names], s["d_radiance"])
        return dict(radiance=B.detach(), **{"d_" + k: v for k, v in zip(names, g)})
    if kind == "envmap":
        return dict(light=project_envmap(s["env"], s["bands"]))
    image, _ = rasterize(s["vertices"], s["radiance"], s["faces"], s["proj"], *s["size"])
    d_v, d_r = torch.autograd.grad(image, [s["vertices"], s["radiance"]], s["d_image"])
    return dict(image=image.detach(), d_vertices=d_v, d_radiance=d_r)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _product_flops(n):
    """One truncated SH product (or square): the Gaunt contraction (about
    353 (K / 16)^2.6 terms) or a separable quadrature, whichever is less."""
    K, QZ, QP = n * n, 3 * (n - 1) // 2 + 1, 3 * (n - 1) + 1
    return min(2.0 * 353.0 * (K / 16.0) ** 2.6, QZ * (4.0 * K + (2 * n - 1) * QP))


def _shade_work(P, N, n, k, fwd_pairs, bwd, saved_in, saved_out):
    K, prod = n * n, _product_flops(n)
    flops = P * ((N * (4.0 * K + 5 * n + 14) if fwd_pairs else 0.0) + (k + 1) * prod + 10 * K)
    read, write = 24.0 + (12.0 if fwd_pairs else 0.0), 12.0
    if saved_in:
        read += 4.0 * (K + 1)
    if saved_out:
        write += 4.0 * (K + 1)
    if bwd:
        flops += P * (N * (9.0 * K + 10 * n + 50) + (2 * k + 3) * prod + 18 * K)
        read += 12.0 + 4.0 * (K + 1)
        write += 12.0
    return flops, P * (read + write)


def _squarings(case):
    return case["fixed_k"] if case.get("fixed_k", -1) >= 0 else 2 if case.get("exp_mode", 0) else 3


def work(case):
    kind = case["kind"]
    if kind in ("step", "render", "relight"):
        f, b = _shade_work(case["points"], case["spheres"], case["bands"], _squarings(case), kind != "relight",
                           kind == "step", kind == "relight", kind == "step")
        return {"flops": f, "bytes": b}
    if kind == "serve":
        f = b = 0.0
        for j in range(case["jobs"]):
            df, db = _shade_work(_rank_points(case, j), _rank_spheres(case, j), 4 if j % 2 else 6, 3, True,
                                 j % 3 != 2, False, True)
            f, b = f + df, b + db
        return {"flops": f, "bytes": b}
    if kind == "views":
        M, V, D = case["theta"] * case["phi"], case["views"], case["params"]
        f, b = _shade_work(M * V, case["spheres"], case["bands"], case["fixed_k"], True, True, False, True)
        rows = 2 * M + case["spheres"]
        return {"flops": f + rows * 12.0 * D + rows * V * 60.0,
                "bytes": b + rows * 2 * 12.0 * D + rows * V * 24.0 + M * V * 24.0}
    if kind == "envmap":
        px = case["height"] * case["width"]
        return {"flops": px * (6.0 * (2 * case["bands"] - 1)) / 4, "bytes": px * 12.0}
    M, px = case["theta"] * case["phi"], case["height"] * case["width"]
    return {"flops": px * 150.0 + 2 * M * 60.0, "bytes": px * (12.0 + 4.0 + 12.0 + 4.0) + M * (12.0 * 6 + 24.0)}


# ---------------------------------------------------------------------------
# float64 restatement
# ---------------------------------------------------------------------------

def _sh_factors(n, z):
    """Per order m, the list over l >= m of N_lm P_lm(z) / sin^m (torch)."""
    out = []
    for m in range(n):
        row, dfact = [], 1.0
        for t in range(1, 2 * m, 2):
            dfact *= t
        p1, p0 = torch.full_like(z, dfact), None
        for l in range(m, n):
            if l == m + 1:
                p0, p1 = p1, (2 * m + 1) * z * p1
            elif l > m + 1:
                p0, p1 = p1, ((2 * l - 1) * z * p1 - (l + m - 1) * p0) / (l - m)
            norm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            row.append((norm * (math.sqrt(2.0) if m else 1.0)) * p1)
        out.append(row)
    return out


def _azimuth(n, x, y):
    c, s = [torch.ones_like(x)], [torch.zeros_like(x)]
    for m in range(1, n):
        c, s = c + [x * c[-1] - y * s[-1]], s + [x * s[-1] + y * c[-1]]
    return c, s


def _sh(n, x, y, z):
    """Real SH [..., n^2]."""
    q, (c, s) = _sh_factors(n, z), _azimuth(n, x, y)
    cols = []
    for l in range(n):
        for m in range(-l, l + 1):
            a = abs(m)
            cols.append(q[a][l - a] * (s[a] if m < 0 else c[a]))
    return torch.stack(cols, -1)


def _rule(nodes, azimuths, n):
    """Gauss-Legendre x uniform rule: (Y [Q, K], w [Q])."""
    t, w = np.polynomial.legendre.leggauss(nodes)
    phi = 2 * np.pi * (np.arange(azimuths) + 0.5) / azimuths
    st = np.sqrt(1 - t * t)
    grid = lambda v: torch.from_numpy(np.ascontiguousarray(v).reshape(-1)).to(DEV)
    x, y, z = grid(st[:, None] * np.cos(phi)), grid(st[:, None] * np.sin(phi)), grid(t[:, None] + 0 * phi)
    return _sh(n, x, y, z), grid(w[:, None] * (2 * np.pi / azimuths) + 0 * phi)


def _log_visibility(n, x, normals, centers, radii, cull):
    d = centers[None] - x[:, None]
    D2 = (d * d).sum(-1)
    invD = D2.rsqrt()
    ratio = radii[None] ** 2 / D2
    open_ = ratio < 1
    s2 = torch.where(open_, ratio, torch.ones_like(ratio))
    c = torch.where(open_, torch.sqrt(torch.where(open_, 1 - ratio, torch.ones_like(ratio))), torch.zeros_like(ratio))
    s = d * invD[..., None]
    q, (ca, sa) = _sh_factors(n, s[..., 2]), _azimuth(n, s[..., 0], s[..., 1])
    keep = None
    if cull:
        u = normals / normals.norm(dim=1, keepdim=True)
        keep = ((d * u[:, None]).sum(-1) >= -radii[None]).to(d.dtype)
    f = [None] * (n * n)
    for l in range(n):
        # int_c^1 P_l(t) dt = (1 - c^2) P_l'(c) / (l (l + 1)), 1 - c for l = 0
        if l == 0:
            G = s2 / (1 + c)
        else:
            G = s2 * _d_legendre(l, c) / (l * (l + 1))
        G = G * (-2 * math.pi * EPSILON)
        if keep is not None:
            G = G * keep
        for m in range(l + 1):
            w = G * q[m][l - m]
            f[l * l + l + m] = (w * ca[m]).sum(1)
            if m:
                f[l * l + l - m] = (w * sa[m]).sum(1)
    return torch.stack(f, 1)


def _d_legendre(l, c):
    """P_l'(c)."""
    p, dp = [torch.ones_like(c), c], [torch.zeros_like(c), torch.ones_like(c)]
    for k in range(1, l):
        p.append(((2 * k + 1) * c * p[k] - k * p[k - 1]) / (k + 1))
        dp.append(dp[k - 1] + (2 * k + 1) * p[k])
    return dp[l]


class _Tail:
    """Float64 exponential and shading of one configuration."""

    def __init__(self, bands, exp_mode, fixed_k):
        self.n, self.mode, self.k = bands, exp_mode, fixed_k
        self.Y, self.w = _rule(3 * (bands - 1) // 2 + 1, 3 * (bands - 1) + 1, bands)
        if exp_mode == 1:
            self.EY, self.Ew = _rule(2 * bands, 4 * bands, bands)
        t, wt = np.polynomial.legendre.leggauss(32)
        t, wt = (t + 1) / 2, wt / 2
        self.ahat = [2 * math.pi * float((wt * t * np.polynomial.legendre.Legendre.basis(l)(t)).sum())
                     for l in range(bands)]

    def mul(self, a, b):
        return ((a @ self.Y.T) * (b @ self.Y.T)) @ (self.w[:, None] * self.Y)

    def visibility(self, f):
        e0 = torch.exp(f[:, :1] / math.sqrt(4 * math.pi))
        g = torch.cat([torch.zeros_like(f[:, :1]), f[:, 1:]], 1)
        if self.mode == 1:
            return e0 * (torch.exp(g @ self.EY.T) @ (self.Ew[:, None] * self.EY))
        with torch.no_grad():
            if self.k >= 0:
                k = torch.full((f.shape[0],), self.k, device=DEV)
            else:
                k = torch.zeros(f.shape[0], device=DEV, dtype=torch.int64)
                n2, thr = (g * g).sum(1), torch.ones((), device=DEV, dtype=torch.float64)
                for _ in range(16):
                    k, thr = k + (n2 > thr), thr * 4
            scale = torch.pow(2.0, -k.to(torch.float64))[:, None]
        g = g * scale
        a = torch.exp((g * g).sum(1, keepdim=True) / (8 * math.pi))
        S = torch.cat([a * math.sqrt(4 * math.pi), a * g[:, 1:]], 1)
        for t in range(int(k.max()) if k.numel() else 0):
            S = torch.where((k > t)[:, None], self.mul(S, S), S)
        return e0 * S

    def radiance(self, f, normals, albedo, light):
        u = normals / normals.norm(dim=1, keepdim=True)
        H = _sh(self.n, u[:, 0], u[:, 1], u[:, 2])
        H = H * torch.tensor([self.ahat[math.isqrt(i)] for i in range(self.n ** 2)], device=DEV, dtype=torch.float64)
        return albedo * (self.mul(self.visibility(f), H) @ light.T)


def _exact_shading(tail, pts, nrm, alb, centers, radii, light, cull, target, dB, wrt):
    """Radiance and, with target (L2) or dB, the loss and the gradients to the
    arrays named in ``wrt`` (points and normals included), in point chunks."""
    P, N = pts.shape[0], centers.shape[0]
    chunk = max(256, min(P, int(1.2e6 / max(N, 8))))
    grad = target is not None or dB is not None
    glob = {k: v.detach().requires_grad_(grad) for k, v in
            dict(centers=centers, radii=radii, light=light).items()}
    out, loss = [], 0.0
    local = {k: [] for k in ("points", "normals", "albedo")}
    for i in range(0, P, chunk):
        loc = {k: v[i:i + chunk].detach().requires_grad_(grad) for k, v in
               dict(points=pts, normals=nrm, albedo=alb).items()}
        f = _log_visibility(tail.n, loc["points"], loc["normals"] if not grad else loc["normals"].detach(),
                            glob["centers"], glob["radii"], cull)
        B = tail.radiance(f, loc["normals"], loc["albedo"], glob["light"])
        out.append(B.detach())
        if grad:
            d = B.detach() - target[i:i + chunk] if target is not None else dB[i:i + chunk]
            loss += 0.5 * float((d * d).sum())
            B.backward(d)
            for k in local:
                local[k].append(loc[k].grad)
    g = {}
    if grad:
        g = {k: (torch.cat(local[k]) if k in local else glob[k].grad) for k in wrt}
    return torch.cat(out), loss, g


def _f64(s):
    return {k: v.detach().double() for k, v in s.items() if torch.is_tensor(v) and v.is_floating_point()}


def _exact_scene(case, seed):
    s = _f64(_scene(case, seed))
    tail = _Tail(case["bands"], case["exp_mode"], case["fixed_k"])
    names = ("light", "albedo", "centers", "radii")
    step = case["kind"] == "step"
    l2 = step and case["api"] == "l2"
    B, loss, g = _exact_shading(tail, s["points"], s["normals"], s["albedo"], s["centers"], s["radii"], s["light"],
                                case["cull"], s["target"] if l2 else None,
                                s["d_radiance"] if step and not l2 else None, names)
    out = dict(radiance=B, **{"d_" + k: v for k, v in g.items()})
    if l2:
        out["loss"] = loss
    return out


def _exact_serve(case, seed):
    out = []
    for job in _serve_jobs(case, seed):
        s = _f64(job)
        B, loss, g = _exact_shading(_Tail(job["bands"], 0, -1), s["points"], s["normals"], s["albedo"], s["centers"],
                                    s["radii"], s["light"], False, s["target"] if job["op"] == "fwdbwd" else None,
                                    None, ("light", "albedo", "centers", "radii"))
        out.append(dict(radiance=B, **{"d_" + k: v for k, v in g.items()}))
        if job["op"] == "fwdbwd":
            out[-1]["loss"] = loss
    return out


def _exact_views(case, seed):
    s = _f64(_views_inputs(case, seed))
    p, poses = s["p"].requires_grad_(True), s["poses"].requires_grad_(True)
    rest = {k: s[b] + (s[A] @ p) for k, b, A in (("v", "v0", "A_v"), ("n", "n0", "A_n"), ("c", "c0", "A_c"))}
    tail = _Tail(case["bands"], 0, case["fixed_k"])
    B, acc, posed, grads = [], {k: 0.0 for k in ("radii", "light", "albedo")}, [], []
    for v in range(case["views"]):
        w, t = poses[v, :3], poses[v, 3:]
        z = torch.zeros((), device=DEV, dtype=torch.float64)
        R = torch.linalg.matrix_exp(torch.stack([torch.stack([z, -w[2], w[1]]), torch.stack([w[2], z, -w[0]]),
                                                 torch.stack([-w[1], w[0], z])]))
        pv, pn, pc = rest["v"] @ R.T + t, rest["n"] @ R.T, rest["c"] @ R.T + t
        b, _, g = _exact_shading(tail, pv.detach(), pn.detach(), s["albedo"], pc.detach(), s["radii"], s["light"],
                                 False, None, s["d_radiance"][v], ("points", "normals", "centers", "radii", "light",
                                                                   "albedo"))
        B.append(b)
        for k in acc:
            acc[k] = acc[k] + g[k]
        posed += [pv, pn, pc]
        grads += [g["points"], g["normals"], g["centers"]]
    dp, dposes = torch.autograd.grad(posed, [p, poses], grads)
    return dict(radiance=torch.stack(B), d_p=dp, d_poses=dposes, **{"d_" + k: v for k, v in acc.items()})


def _exact_envmap(case, seed):
    env, H, W, n = _env_inputs(case, seed), case["height"], case["width"], case["bands"]
    k = torch.arange(W, device=DEV, dtype=torch.float64)
    phi = (k + 0.5) * (2 * math.pi / W)
    c = torch.stack([torch.cos(m * phi) for m in range(n)] + [torch.sin(m * phi) for m in range(n)], 1)
    mom = torch.cat([torch.einsum("hwc,wf->hcf", env[i:i + 256].double(), c) for i in range(0, H, 256)])
    r = torch.arange(H, device=DEV, dtype=torch.float64)
    th = (r + 0.5) * (math.pi / H)
    area = (torch.cos(r * (math.pi / H)) - torch.cos((r + 1) * (math.pi / H))) * (2 * math.pi / W)
    q, st = _sh_factors(n, torch.cos(th)), torch.sin(th)
    cols = []
    for l in range(n):
        for m in range(-l, l + 1):
            a = abs(m)
            cols.append(((q[a][l - a] * st ** a * area)[:, None] * mom[:, :, a + (n if m < 0 else 0)]).sum(0))
    return dict(light=torch.stack(cols, 1))


def _exact_raster(case, seed):
    s = _raster_inputs(case, seed)
    H, W, faces = case["height"], case["width"], s["faces"].long()
    vert = s["vertices"].double().requires_grad_(True)
    rad = s["radiance"].double().requires_grad_(True)
    P = torch.from_numpy(np.asarray(s["proj"], np.float64)).to(DEV)
    clip = vert @ P[:, :3].T + P[:, 3]
    with torch.no_grad():
        ndc = clip / clip[:, 3:]
        tri = ndc[faces]                                                   # [F, 3, 4]
        ok = (clip[faces][..., 3] > 0).all(1)
        edge = lambda a, b, x, y: (b[:, 0] - a[:, 0]) * (y - a[:, 1]) - (b[:, 1] - a[:, 1]) * (x - a[:, 0])
        area = edge(tri[:, 0], tri[:, 1], tri[:, 2, 0], tri[:, 2, 1])
        c0 = torch.ceil((tri[..., 0].amin(1) + 1) * 0.5 * W - 0.5).clamp(min=0).long()
        c1 = torch.floor((tri[..., 0].amax(1) + 1) * 0.5 * W - 0.5).clamp(max=W - 1).long()
        r0 = torch.ceil((1 - tri[..., 1].amax(1)) * 0.5 * H - 0.5).clamp(min=0).long()
        r1 = torch.floor((1 - tri[..., 1].amin(1)) * 0.5 * H - 0.5).clamp(max=H - 1).long()
        depth = torch.full((H * W,), math.inf, device=DEV, dtype=torch.float64)
        best = torch.full((H * W,), faces.shape[0], device=DEV, dtype=torch.int64)
        ids = torch.arange(faces.shape[0], device=DEV)
        hits = []
        nr, nc = int((r1 - r0)[ok].max()) + 1, int((c1 - c0)[ok].max()) + 1
        for i in range(nr):
            for j in range(nc):
                live = torch.nonzero(ok & (r0 + i <= r1) & (c0 + j <= c1)).flatten()
                if not live.numel():
                    continue
                r, c, t = r0[live] + i, c0[live] + j, tri[live]
                x, y = -1 + (2.0 * c + 1) / W, 1 - (2.0 * r + 1) / H
                lam = torch.stack([edge(t[:, 1], t[:, 2], x, y), edge(t[:, 2], t[:, 0], x, y),
                                   edge(t[:, 0], t[:, 1], x, y)], 1) / area[live, None]
                zz = (lam * t[..., 2]).sum(1)
                m = (lam >= 0).all(1) & (zz >= -1) & (zz <= 1)
                pix, zz = (r * W + c)[m], zz[m]
                depth.scatter_reduce_(0, pix, zz, "amin")
                hits.append((pix, zz, ids[live][m]))
        for pix, zz, f in hits:
            front = zz == depth[pix]
            best.scatter_reduce_(0, pix[front], f[front], "amin")
        seen = torch.nonzero(best < faces.shape[0]).flatten()
    v = faces[best[seen]]
    cl = clip[v]
    n = cl[..., :2] / cl[..., 3:]
    x, y = -1 + (2.0 * (seen % W) + 1) / W, 1 - (2.0 * (seen // W) + 1) / H
    e = torch.stack([edge(n[:, 1], n[:, 2], x, y), edge(n[:, 2], n[:, 0], x, y), edge(n[:, 0], n[:, 1], x, y)], 1)
    u = e / e.sum(1, keepdim=True) / cl[..., 3]
    b = u / u.sum(1, keepdim=True)
    image = torch.zeros((H * W, 3), device=DEV, dtype=torch.float64).index_put((seen,), (b[..., None] * rad[v]).sum(1))
    image = image.reshape(H, W, 3)
    dv, dr = torch.autograd.grad(image, [vert, rad], s["d_image"].double())
    return dict(image=image.detach(), d_vertices=dv, d_radiance=dr)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "render", "relight"):
        return _exact_scene(case, seed)
    return {"serve": _exact_serve, "views": _exact_views, "envmap": _exact_envmap,
            "raster": _exact_raster}[kind](case, seed)

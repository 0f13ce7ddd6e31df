"""The work that users of this renderer have it do, as cases to be timed and checked.

A case is a dict of plain values; `prepare` makes what a program holds before the call (seeded
inputs on the GPU, output buffers, workspaces), `run` is one pass through the public entry points,
`work` what a pass cannot do without and `exact` the same outputs from plain 64-bit torch.

Scenes follow the recipe of the repository's generator (spheres on a ground square, metal or
dielectric, point lights above them, a sky with two suns), made here with torch.  The lighting set of a
frame is made by pooling the environment, as a program would load one from a file, so that a
frame's inputs do not depend on the precompute's rounding.
"""
import math

import numpy as np
import torch

import paper_2012_03325_gb300 as ep

NEAR = 0.05
INF = float("inf")
F64 = torch.float64


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def _frame(w, h, lights, **more):
    c = dict(kind="frame", width=w, height=h, lights=lights, spheres=200, samples=32, env=2048, levels=8,
             compact=False, half=False, colour=False, reinhard=False)
    c.update(more)
    return c


def listed():
    return [
        # a thumbnail or tracking preview: three dependent launches, latency and host time count
        dict(_frame(256, 256, 4, spheres=16, samples=16, env=128, levels=6), name="frame_256"),
        # the everyday frame: 1080p, FP32 G-buffer, 64 white lights, HDR and 8-bit image
        dict(_frame(1920, 1080, 64), name="frame_1080p"),
        # a view of odd size in a tool's viewport: compact G-buffer, few coloured lights
        dict(_frame(1283, 721, 12, compact=True, colour=True, spheres=60, env=1024), name="frame_ragged_colour"),
        # the largest view: 2160p with the compact G-buffer and the FP16 HDR image
        dict(_frame(3840, 2160, 64, compact=True, half=True), name="frame_2160p_compact"),
        # a static scene with per-light shadow maps: shading only, the maps resident
        dict(kind="shadow", width=1920, height=1080, lights=64, size=512, spheres=200, colour=False,
             name="shadow_1080p"),
        # the scene or the lights moved: every light's map rendered again
        dict(kind="maps", lights=64, size=512, spheres=200, lat=16, lon=32, ground=64, name="shadow_maps_64"),
        # a mesh rasterised into the G-buffer each frame
        dict(kind="mesh", width=1920, height=1080, spheres=200, lat=16, lon=32, ground=64, name="mesh_1080p"),
        # a surfel cloud from a SLAM system splatted into the G-buffer each frame
        dict(kind="surfels", width=1920, height=1080, spheres=200, per_sphere=4000, ground=400000, tol=0.01,
             name="surfels_1080p"),
        # bloom over an HDR frame with highlights, tone map fused, HDR kept
        dict(kind="bloom", width=1920, height=1080, levels=6, radius=4, half=False, spots=24, name="bloom_1080p"),
        # a point cloud shaded from its depth
        dict(kind="edl", width=1920, height=1080, radius=1, directions=8, compact=False, half=False,
             name="edl_1080p"),
        # an environment is loaded: the whole lighting set
        dict(kind="ibl", env_w=2048, env_h=1024, levels=8, samples=1024, lut=64, lut_samples=1024, name="ibl_2048"),
        # synthetic training images: many small views in one batch
        dict(kind="batch", views=64, width=256, height=256, spheres=16, samples=32, env=512, levels=7,
             name="batch_64x256"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "shadow", "maps", "mesh", "surfels", "bloom", "edl", "ibl", "batch"])
    flag = lambda: rng.random() < 0.5
    if kind == "frame":
        env = rng.choice([128, 256, 512, 1024, 2048])
        return _frame(_log(rng, 96, 3840), _log(rng, 64, 2160), _log(rng, 1, 256), spheres=_log(rng, 8, 200),
                      samples=rng.choice([8, 16, 24, 32, 64]), env=env, levels=rng.randint(5, 8), compact=flag(),
                      half=flag(), colour=rng.random() < 0.3, reinhard=rng.random() < 0.3)
    if kind == "shadow":
        return dict(kind=kind, width=_log(rng, 128, 1920), height=_log(rng, 96, 1080), lights=_log(rng, 1, 64),
                    size=_log(rng, 96, 768), spheres=_log(rng, 8, 200), colour=rng.random() < 0.3)
    if kind == "maps":
        return dict(kind=kind, lights=_log(rng, 1, 64), size=_log(rng, 64, 1024), spheres=_log(rng, 8, 200),
                    lat=rng.randint(6, 18), lon=rng.randint(8, 32), ground=rng.randint(4, 96))
    if kind == "mesh":
        return dict(kind=kind, width=_log(rng, 128, 2560), height=_log(rng, 96, 1440), spheres=_log(rng, 4, 200),
                    lat=rng.randint(6, 18), lon=rng.randint(8, 32), ground=rng.randint(2, 96))
    if kind == "surfels":
        return dict(kind=kind, width=_log(rng, 128, 2560), height=_log(rng, 96, 1440), spheres=_log(rng, 4, 200),
                    per_sphere=_log(rng, 200, 4000), ground=_log(rng, 2000, 400000), tol=rng.choice([0.0, 0.01, 0.05]))
    if kind == "bloom":
        return dict(kind=kind, width=_log(rng, 96, 3840), height=_log(rng, 64, 2160), levels=rng.randint(2, 6),
                    radius=rng.randint(1, 8), half=flag(), spots=_log(rng, 4, 60))
    if kind == "edl":
        return dict(kind=kind, width=_log(rng, 96, 3840), height=_log(rng, 64, 2160), radius=rng.randint(1, 4),
                    directions=rng.choice([4, 8, 8, 12]), compact=flag(), half=flag())
    if kind == "ibl":
        w = _log(rng, 96, 2048)
        return dict(kind=kind, env_w=w, env_h=max(32, w // 2 + rng.choice([0, 0, 0, 1, 7])), levels=rng.randint(3, 8),
                    samples=_log(rng, 64, 1024), lut=rng.choice([16, 32, 48, 64]), lut_samples=_log(rng, 64, 1024))
    return dict(kind="batch", views=rng.randint(4, 64), width=_log(rng, 64, 512), height=_log(rng, 64, 512),
                spheres=rng.randint(8, 32), samples=rng.choice([16, 32]), env=rng.choice([128, 256, 512]),
                levels=rng.randint(5, 7))


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50.0)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


def work(case):
    """Inputs read once, outputs written once; FLOP of the method (see each line)."""
    k = case["kind"]
    if k == "ibl":
        n0 = case["env_w"] * case["env_h"]
        texels = sum(max(1, case["env_w"] >> m) * max(1, case["env_h"] >> m) for m in range(1, case["levels"]))
        # four taps of three channels per prefiltered texel and sample; a table entry's sample ~40
        return {"bytes": 16.0 * (2 * n0 + texels + 512) + 8.0 * case["lut"] ** 2,
                "flops": 24.0 * texels * case["samples"] + 40.0 * case["lut"] ** 2 * case["lut_samples"]}
    if k == "maps":
        v, t = _mesh_counts(case)
        n = case["lights"]
        return {"bytes": 48.0 * v + 12.0 * t + 4.0 * n * case["size"] ** 2, "flops": n * (120.0 * t + 30.0 * case["size"] ** 2)}
    px = case["width"] * case["height"]
    if k == "mesh":
        v, t = _mesh_counts(case)
        return {"bytes": 48.0 * v + 12.0 * t + 40.0 * px, "flops": 120.0 * t + 90.0 * px}
    if k == "surfels":
        n = case["spheres"] * case["per_sphere"] + _side(case["ground"]) ** 2
        return {"bytes": 64.0 * n + 40.0 * px, "flops": 250.0 * n + 6.5 * 45.0 * px}
    hdr = 8.0 if case.get("half") else 16.0
    if k == "bloom":
        return {"bytes": px * (2 * hdr + 4.0), "flops": px * (36.0 + 90.0 + 4.0 * case["radius"])}
    if k == "edl":
        return {"bytes": px * (4.0 + (4.0 if case["compact"] else 16.0) + hdr + 4.0),
                "flops": px * (40.0 + 3.0 * case["directions"])}
    if k == "batch":
        px *= case["views"]
        lights, env = 64.0, 8.0  # the views' mean light count
    else:
        lights, env = case["lights"], 16.0
    g = 14.0 if case.get("compact") else 36.0
    # about three quarters of a view is surface; 85 FLOP per surface pixel and light, 300 per pixel
    flops = px * (0.75 * 85.0 * lights + 300.0)
    if k == "shadow":
        return {"bytes": px * (g + 20.0) + 4.0 * lights * case["size"] ** 2, "flops": flops + px * 0.75 * 40.0 * lights}
    return {"bytes": px * (g + hdr + 4.0) + env, "flops": flops + px / 4 * (30.0 * case["samples"] + 490.0)}


def _side(ground):
    return max(1, int(round(math.sqrt(ground))))


def _mesh_counts(case):
    la, lo, s, g = case["lat"], case["lon"], case["spheres"], case["ground"]
    return s * (la + 1) * lo + (g + 1) ** 2, s * 2 * lo * (la - 1) + 2 * g * g


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _look_at(eye, target, up=(0.0, 1.0, 0.0)):
    eye = np.asarray(eye, np.float64)
    f = np.asarray(target, np.float64) - eye
    f /= np.linalg.norm(f)
    r = np.cross(f, np.asarray(up, np.float64))
    r /= np.linalg.norm(r)
    m = np.eye(4)
    m[:3, 0], m[:3, 1], m[:3, 2], m[:3, 3] = r, np.cross(r, f), -f, eye
    return m


class _Scene:
    def __init__(self, seed, spheres, lights=1, colour=False):
        g = np.random.default_rng(seed)
        self.F = F = 5.0 * math.sqrt(spheres / 16.0)
        self.r = g.uniform(0.2, 1.0, spheres)
        self.c = np.stack([g.uniform(-F, F, spheres), self.r, g.uniform(-F, F, spheres)], 1)
        n = spheres + 1  # the last one is the ground's material
        self.albedo = g.uniform(0.0, 1.0, (n, 3))
        self.metal = (g.uniform(size=n) < 0.5).astype(np.float64)
        self.rough = g.uniform(0.05, 1.0, n)
        self.lights = np.zeros((lights, 8), np.float32)
        self.lights[:, 0] = g.uniform(-F, F, lights)
        self.lights[:, 1] = g.uniform(3.0, 3.0 + 2.0 * F, lights)
        self.lights[:, 2] = g.uniform(-F, F, lights)
        self.lights[:, 3] = g.uniform(1.0, 50.0, lights)
        self.lights[:, 4:7] = g.uniform(0.2, 1.0, (lights, 3)) if colour else 1.0
        self.half = 8.0 * F
        self.view = _look_at((0.0, 0.6 * F, 1.6 * F), (0.0, 0.0, 0.0))
        self.fov = math.radians(60.0)
        self.g = g


def _t(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _cast(sc, W, H, view=None, fov=None, want_normals=True):
    """(depth, material index, normal) of every pixel centre's ray, in 64 bits."""
    view, fov = sc.view if view is None else view, sc.fov if fov is None else fov
    t = math.tan(0.5 * fov)
    px = (2.0 * (torch.arange(W, device="cuda", dtype=F64) + 0.5) / W - 1.0) * t * W / H
    py = (1.0 - 2.0 * (torch.arange(H, device="cuda", dtype=F64) + 0.5) / H) * t
    px, py = px[None, :].expand(H, W).reshape(-1), py[:, None].expand(H, W).reshape(-1)
    R, eye = view[:3, :3], view[:3, 3]
    d = [R[i, 0] * px + R[i, 1] * py - R[i, 2] for i in range(3)]
    tp = torch.where(d[1] < 0, -eye[1] / d[1], INF)
    hit = torch.isfinite(tp) & (tp > 0) & ((eye[0] + tp * d[0]).abs() <= sc.half) & ((eye[2] + tp * d[2]).abs() <= sc.half)
    best = torch.where(hit, tp, INF)
    n = len(sc.r)
    mat = torch.where(hit, n, -1)
    a = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    step = max(1, (1 << 25) // (W * H))
    for s in range(0, n, step):
        o = _t(eye[None, :] - sc.c[s:s + step], F64)
        b = o[:, 0:1] * d[0] + o[:, 1:2] * d[1] + o[:, 2:3] * d[2]
        disc = b * b - a * ((o * o).sum(1) - _t(sc.r[s:s + step], F64) ** 2)[:, None]
        th = torch.where(disc >= 0, (-b - disc.clamp_min(0).sqrt()) / a, INF)
        th = torch.where(th > 1e-6, th, INF)
        th, k = th.min(0)
        take = th < best
        best, mat = torch.where(take, th, best), torch.where(take, k + s, mat)
    if not want_normals:
        return best.view(H, W), None, None
    c = torch.cat([_t(sc.c, F64), torch.zeros(1, 3, device="cuda", dtype=F64)])[mat.clamp_min(0)]
    e = best.where(mat >= 0, torch.ones_like(best))
    nrm = torch.stack([eye[i] + e * d[i] - c[:, i] for i in range(3)], 1)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    nrm[mat == n] = torch.tensor([0.0, 1.0, 0.0], device="cuda", dtype=F64)
    nrm[mat < 0] = 0.0
    return best.view(H, W), mat.view(H, W), nrm.view(H, W, 3)


def _planes(sc, W, H, compact):
    """The render targets of the ray-cast scene in the FP32 or the compact layout."""
    depth, mat, nrm = _cast(sc, W, H)
    on = mat >= 0
    m = mat.clamp_min(0)
    alb = _t(sc.albedo, F64)[m] * on[..., None]
    met, rough = _t(sc.metal, F64)[m] * on, _t(sc.rough, F64)[m] * on
    depth = depth.float()
    if not compact:
        return [torch.cat([alb, met[..., None]], 2).float(), torch.cat([nrm, rough[..., None]], 2).float(), depth]
    srgb = torch.where(alb <= 0.0031308, 12.92 * alb, 1.055 * alb.clamp_min(1e-9) ** (1 / 2.4) - 0.055)
    rt0 = torch.cat([torch.floor(255.0 * srgb + 0.5), torch.full_like(met[..., None], 255.0)], 2).to(torch.uint8)
    s = nrm.abs().sum(2, keepdim=True)
    p = nrm[..., :2] / torch.where(s == 0, 1.0, s)
    fold = (1.0 - p.flip(2).abs()) * torch.where(p >= 0, 1.0, -1.0)
    rt1 = torch.where(nrm[..., 2:] < 0, fold, p).half()
    rt2 = torch.stack([torch.floor(255.0 * met + 0.5), torch.floor(255.0 * rough + 0.5)], 2).to(torch.uint8)
    return [rt0, rt1.contiguous(), rt2, depth]


def _sky(seed, W, H):
    g = np.random.default_rng(seed + 77)
    phi = 2 * math.pi * ((torch.arange(W, device="cuda", dtype=F64) + 0.5) / W - 0.5)
    th = math.pi * (torch.arange(H, device="cuda", dtype=F64) + 0.5) / H
    d = torch.stack([th.sin()[:, None] * phi.sin(), th.cos()[:, None].expand(H, W), -th.sin()[:, None] * phi.cos()], 2)
    t = 0.5 * (d[..., 1:2] + 1.0)
    lo, hi = _t([0.3, 0.25, 0.2], F64), _t([0.25, 0.45, 0.9], F64)
    col = lo + (hi - lo) * t
    for _ in range(2):
        el, az, sig = math.radians(g.uniform(10, 70)), g.uniform(0, 2 * math.pi), math.radians(g.uniform(2, 6))
        sun = _t([math.cos(el) * math.sin(az), math.sin(el), -math.cos(el) * math.cos(az)], F64)
        a = torch.arccos(((d * sun).sum(2)).clamp(-1, 1))
        col = col + 100.0 * torch.exp(-a * a / (2 * sig * sig))[..., None]
    return torch.cat([col, torch.ones_like(t)], 2).float().contiguous()


def _maps_of(seed, env_w, levels):
    """A lighting set (levels, irradiance, table) of plain tensors: the pooled sky."""
    sky = _sky(seed, env_w, env_w // 2)
    img = sky.permute(2, 0, 1)[None]
    pool = torch.nn.functional.adaptive_avg_pool2d
    lev = [sky]
    for m in range(1, levels):
        lev.append(pool(img, (max(1, (env_w // 2) >> m), max(1, env_w >> m)))[0].permute(1, 2, 0).contiguous())
    coarse = pool(img, (4, 8))
    irr = torch.nn.functional.interpolate(coarse, size=(16, 32), mode="bilinear")[0].permute(1, 2, 0).contiguous()
    x = (torch.arange(64, device="cuda", dtype=torch.float32) + 0.5) / 64
    mu, r = x[None, :].expand(64, 64), x[:, None].expand(64, 64)
    # a rational fit of the split-sum table's shape
    a = (1.0 - r) * (0.3 + 0.7 * mu) + r * (0.15 + 0.4 * mu)
    lut = torch.stack([a * 0.95, (1.0 - mu) ** 4 * 0.3 * (1.0 - 0.7 * r)], 2).contiguous()
    return lev, irr, lut


def _lighting(maps, env_w, levels):
    lev, irr, lut = maps
    ibl = ep.Ibl(ep.ibl_params(levels, 1, 64, 1, 32, 16), env_w, env_w // 2)
    for m in range(levels):
        ibl.level(m).copy_(lev[m])
    ibl.irradiance().copy_(irr)
    ibl.lut().copy_(lut)
    return ibl


def _ssao_inputs(seed, K):
    g = np.random.default_rng(seed + 11)
    v = np.stack([g.uniform(-1, 1, K), g.uniform(-1, 1, K), g.uniform(0.05, 1, K)], 1)
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    v *= (g.uniform(size=K) * (0.1 + 0.9 * (np.arange(K) / K) ** 2))[:, None]
    phi = g.uniform(0, 2 * math.pi, 16)
    return _t(np.concatenate([v, np.zeros((K, 1))], 1)), _t(np.stack([np.cos(phi), np.sin(phi)], 1))


def _camera(sc, W, H):
    return ep.camera(sc.view.astype(np.float32).T.reshape(-1), sc.fov, W, H)


def _gbuffer(planes):
    return ep.GBuffer.compact(*planes) if len(planes) == 4 else ep.GBuffer.fp32(*planes)


def _out(H, W, half=False, n=None):
    lead = () if n is None else (n,)
    hdr = torch.zeros(*lead, H, W, 4, device="cuda", dtype=torch.float16 if half else torch.float32)
    return hdr, torch.zeros(*lead, H, W, 4, device="cuda", dtype=torch.uint8)


def _tone(case):
    return ep.tonemap_params(1.0, ep.EPBR_TONEMAP_REINHARD if case.get("reinhard") else ep.EPBR_TONEMAP_ACES)


def _mesh(sc, lat, lon, cells):
    th, ph = np.linspace(0, math.pi, lat + 1), np.linspace(0, 2 * math.pi, lon + 1)[:-1]
    T, P = np.meshgrid(th, ph, indexing="ij")
    nrm = np.stack([np.sin(T) * np.cos(P), np.cos(T), np.sin(T) * np.sin(P)], -1).reshape(-1, 3)
    i, j = np.meshgrid(np.arange(lat), np.arange(lon), indexing="ij")
    a, b, c, d = i * lon + j, i * lon + (j + 1) % lon, (i + 1) * lon + j, (i + 1) * lon + (j + 1) % lon
    q = np.concatenate([np.stack([a, c, b], -1)[1:].reshape(-1, 3), np.stack([b, c, d], -1)[:-1].reshape(-1, 3)])
    S, n = len(sc.r), len(nrm)
    v = np.zeros((S, n, 12))
    v[:, :, 0:3] = sc.c[:, None] + sc.r[:, None, None] * nrm
    v[:, :, 3:6] = nrm
    v[:, :, 6:9], v[:, :, 9], v[:, :, 10] = sc.albedo[:S, None], sc.metal[:S, None], sc.rough[:S, None]
    k = cells + 1
    X, Z = np.meshgrid(np.linspace(-sc.half, sc.half, k), np.linspace(-sc.half, sc.half, k), indexing="ij")
    gv = np.zeros((k * k, 12))
    gv[:, 0], gv[:, 2], gv[:, 4] = X.reshape(-1), Z.reshape(-1), 1.0
    gv[:, 6:9], gv[:, 9], gv[:, 10] = sc.albedo[-1], sc.metal[-1], sc.rough[-1]
    idx = np.arange(k * k).reshape(k, k)
    a, b, c, d = (x.reshape(-1) for x in (idx[:-1, :-1], idx[1:, :-1], idx[:-1, 1:], idx[1:, 1:]))
    gt = np.stack([np.stack([a, b, c], 1), np.stack([b, d, c], 1)], 1).reshape(-1, 3) + S * n
    tri = np.concatenate([(q[None] + (np.arange(S) * n)[:, None, None]).reshape(-1, 3), gt])
    return _t(np.concatenate([v.reshape(-1, 12), gv])), _t(tri, torch.int32)


def _surfels(sc, per_sphere, ground, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=F64)
    ru = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=F64)
    S, side = len(sc.r), _side(ground)
    n = rn(S, per_sphere, 3)
    n = n / n.norm(dim=2, keepdim=True)
    r = _t(sc.r, F64)[:, None, None]
    cell = 2.0 * sc.half / side
    x = (torch.arange(side, device="cuda", dtype=F64) + 0.5) * cell - sc.half
    gp = torch.stack([x[:, None].expand(side, side), torch.zeros(side, side, device="cuda", dtype=F64),
                      x[None, :].expand(side, side)], 2).reshape(-1, 3)
    gp[:, 0] += (ru(side * side) - 0.5) * 0.6 * cell
    gp[:, 2] += (ru(side * side) - 0.5) * 0.6 * cell
    P = torch.cat([(_t(sc.c, F64)[:, None] + r * n).reshape(-1, 3), gp])
    N = torch.cat([n.reshape(-1, 3), torch.tensor([[0.0, 1.0, 0.0]], device="cuda", dtype=F64).expand(side * side, 3)])
    space = torch.cat([(4 * math.pi * r[:, :, 0] ** 2 / per_sphere).sqrt().expand(S, per_sphere).reshape(-1),
                       torch.full((side * side,), cell, device="cuda", dtype=F64)])
    k = torch.cat([torch.arange(S, device="cuda").repeat_interleave(per_sphere),
                   torch.full((side * side,), S, device="cuda")])
    m = len(P)
    t = rn(m, 3)
    t = t - N * (t * N).sum(1, keepdim=True)
    t = t / t.norm(dim=1, keepdim=True)
    a = 1.2 * space * (0.8 + 0.4 * ru(m))
    b = a * (0.6 + 0.4 * ru(m))
    alb = (_t(sc.albedo, F64)[k] + 0.1 * (ru(m, 3) - 0.5)).clamp(0, 1)
    col = lambda v: v[:, None]
    rec = torch.cat([P, col(a), N, col(b), t, col(_t(sc.metal, F64)[k]), alb, col(_t(sc.rough, F64)[k])], 1)
    return rec.float().contiguous()


def _hdr_field(case, seed):
    """A smooth frame below the bloom threshold with bright discs and single bright pixels."""
    W, H = case["width"], case["height"]
    g = np.random.default_rng(seed)
    gt = torch.Generator(device="cuda").manual_seed(seed)
    x, y = torch.arange(W, device="cuda", dtype=torch.float32)[None], torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    base = 0.8 * (0.5 * x / W + 0.3 * y / H + 0.2 * torch.rand(H, W, generator=gt, device="cuda"))
    img = base[..., None] * _t([1.0, 0.9, 0.8, 0.0])
    for _ in range(case["spots"]):
        cx, cy, r = g.uniform(0, W), g.uniform(0, H), g.uniform(1, 24)
        x0, x1, y0, y1 = max(0, int(cx - r)), min(W, int(cx + r) + 2), max(0, int(cy - r)), min(H, int(cy + r) + 2)
        sub = img[y0:y1, x0:x1]
        in_ = (x[:, x0:x1] - cx) ** 2 + (y[y0:y1] - cy) ** 2 <= r * r
        img[y0:y1, x0:x1] = torch.where(in_[..., None], _t(g.uniform(2, 60, 4)), sub)
    n = max(1, W * H // 4096)
    img[_t(g.integers(0, H, n), torch.long), _t(g.integers(0, W, n), torch.long)] = _t(g.uniform(2, 100, 4))
    img[..., 3] = 1.0
    return (img.half() if case["half"] else img).contiguous()


def _cloud(case, seed):
    """A point cloud's colour and depth: rough layers, splatted over about 70% of the image."""
    W, H = case["width"], case["height"]
    g = np.random.default_rng(seed)
    gt = torch.Generator(device="cuda").manual_seed(seed)
    x, y = torch.arange(W, device="cuda", dtype=torch.float32)[None], torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    depth = torch.full((H, W), INF, device="cuda")
    col = torch.zeros(H, W, 3, device="cuda")
    for _ in range(4):
        z = g.uniform(2, 40) * (1 + 0.1 * torch.sin(x / g.uniform(5, 30)) * torch.cos(y / g.uniform(5, 30)))
        z = z * (1 + 0.02 * (2 * torch.rand(H, W, generator=gt, device="cuda") - 1))
        keep = (torch.rand(H, W, generator=gt, device="cuda") < 0.35) & (z < depth)
        depth = torch.where(keep, z, depth)
        c = _t(g.uniform(0.05, 1.0, 3)) * (0.7 + 0.3 * torch.rand(H, W, 1, generator=gt, device="cuda"))
        col = torch.where(keep[..., None], c, col)
    zero = torch.zeros(H, W, 1, device="cuda")
    if case["compact"]:
        rt0 = torch.cat([torch.floor(255 * col.clamp(0, 1) ** (1 / 2.2) + 0.5), zero + 255], 2).to(torch.uint8)
        return [rt0, torch.zeros(H, W, 2, device="cuda", dtype=torch.float16),
                torch.zeros(H, W, 2, device="cuda", dtype=torch.uint8), depth]
    return [torch.cat([col, zero], 2).contiguous(), torch.zeros(H, W, 4, device="cuda"), depth]


def _light_cameras(sc):
    views = []
    for p in sc.lights[:, :3].astype(np.float64):
        f = -p / np.linalg.norm(p)
        views.append(_look_at(p, (0, 0, 0), (0.0, 0.0, -1.0) if abs(f[2]) < 0.9 else (1.0, 0.0, 0.0)))
    return views


def _shadow_inputs(sc, S):
    views = _light_cameras(sc)
    maps = torch.stack([_cast(sc, S, S, v, math.radians(90.0), False)[0].float() for v in views])
    cams = np.zeros((len(views), 16), np.float32)
    for i, v in enumerate(views):
        cams[i, :12] = np.linalg.inv(v)[:3, :4].reshape(-1)
        cams[i, 12] = 1.0 / math.tan(math.radians(45.0))
    return maps.contiguous(), _t(cams)


def _batch_lights(case, seed):
    g = np.random.default_rng(seed + 5)
    return [int(round(math.exp(g.uniform(math.log(16), math.log(256))))) for _ in range(case["views"])]


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k, "case": case}
    if k == "ibl":
        s["env"] = _sky(seed, case["env_w"], case["env_h"])
        p = ep.ibl_params(case["levels"], case["samples"], case["lut"], case["lut_samples"], 32, 16)
        s["ibl"] = ep.Ibl(p, case["env_w"], case["env_h"])
        n = ep.epbr_precompute_ibl_workspace_size(p, case["env_w"], case["env_h"])
        s["ws"] = torch.empty(n + 512, dtype=torch.uint8, device="cuda")
        return s
    if k == "maps":
        sc = _Scene(seed, case["spheres"], case["lights"])
        S = case["size"]
        s["mesh"] = ep.Mesh(*_mesh(sc, case["lat"], case["lon"], case["ground"]))
        s["cams"] = [ep.camera(v.astype(np.float32).T.reshape(-1), math.radians(90.0), S, S) for v in _light_cameras(sc)]
        s["maps"] = torch.zeros(case["lights"], S, S, device="cuda")
        n = ep.epbr_shadow_maps_workspace_size(s["mesh"].struct.num_triangles, S)
        s["ws"] = torch.empty(n + 512, dtype=torch.uint8, device="cuda")
        return s
    W, H = case["width"], case["height"]
    if k in ("mesh", "surfels"):
        sc = _Scene(seed, case["spheres"])
        s["cam"] = _camera(sc, W, H)
        s["rt"] = [torch.zeros(H, W, 4, device="cuda"), torch.zeros(H, W, 4, device="cuda"), torch.zeros(H, W, device="cuda")]
        s["gb"] = ep.GBuffer.fp32(*s["rt"])
        if k == "mesh":
            s["mesh"] = ep.Mesh(*_mesh(sc, case["lat"], case["lon"], case["ground"]))
            s["ids"] = torch.zeros(H, W, dtype=torch.int32, device="cuda")
            n = ep.epbr_raster_workspace_size(s["mesh"].struct.num_triangles, W, H)
        else:
            s["surfels"] = ep.Surfels(_surfels(sc, case["per_sphere"], case["ground"], seed))
            s["weight"] = torch.zeros(H, W, device="cuda")
            n = ep.epbr_surfel_workspace_size(s["surfels"].struct.num_surfels, W, H)
        s["ws"] = torch.empty(n + 512, dtype=torch.uint8, device="cuda")
        return s
    s["tp"] = _tone(case)
    half = bool(case.get("half"))
    s["fmt"] = ep.EPBR_HDR_RGBA16F if half else ep.EPBR_HDR_RGBA32F
    if k == "batch":
        n = case["views"]
        s["hdr"], s["ldr"] = _out(H, W, False, n)
        maps = [_maps_of(seed + e, case["env"], case["levels"]) for e in range(2)]
        s["ibls"] = [_lighting(m, case["env"], case["levels"]) for m in maps]
        kern, noise = _ssao_inputs(seed, case["samples"])
        s["ssao"] = ep.SsaoParams(kern, noise, radius=0.5)
        views, keep = [], []
        for v, nl in enumerate(_batch_lights(case, seed)):
            sc = _Scene(seed * 1000 + v, case["spheres"], nl)
            gb, lights = _gbuffer(_planes(sc, W, H, False)), _t(sc.lights)
            keep += [gb, lights]
            views.append(ep.view(gb, _camera(sc, W, H), lights, v % 2, s["ldr"][v], s["hdr"][v]))
        s["batch"] = ep.Batch(views, s["ibls"], ep.batch_params(s["ssao"], tp=s["tp"]), keep=keep)
        s["batch"].set_plan(1)  # the staged plan, which the autotuner keeps on small views
        return s
    if k == "bloom":
        s["src"] = _hdr_field(case, seed)
        s["hdr"], s["ldr"] = _out(H, W, half)
        s["bp"] = ep.bloom_params(1.0, 0.5, 2.0, case["radius"], case["levels"])
        s["ws"] = torch.empty(ep.epbr_bloom_workspace_size(W, H, s["bp"]) + 512, dtype=torch.uint8, device="cuda")
        return s
    if k == "edl":
        s["gb"] = _gbuffer(_cloud(case, seed))
        s["hdr"], s["ldr"] = _out(H, W, half)
        s["ep"] = ep.edl_params(8.0, case["radius"], case["directions"])
        return s
    sc = _Scene(seed, case["spheres"], case["lights"], case["colour"])
    env_w, levels = case.get("env", 1024), case.get("levels", 8)
    s["gb"] = _gbuffer(_planes(sc, W, H, bool(case.get("compact"))))
    s["cam"], s["lights"] = _camera(sc, W, H), _t(sc.lights)
    s["ibl"] = _lighting(_maps_of(seed, env_w, levels), env_w, levels)
    s["hdr"], s["ldr"] = _out(H, W, half)
    if k == "shadow":
        s["shadows"] = ep.Shadows(*_shadow_inputs(sc, case["size"]))
        s["params"] = ep.shade_params()
        return s
    s["ssao"] = ep.SsaoParams(*_ssao_inputs(seed, case["samples"]), radius=0.5)
    ha, wa = s["ssao"].ao_shape(W, H)
    s["ao"] = torch.zeros(ha, wa, device="cuda")
    s["ws"] = torch.empty(4 * ha * wa + 512, dtype=torch.uint8, device="cuda")
    s["params"] = ep.shade_params(ep.EPBR_SHADE_ALL | ep.EPBR_SHADE_EARLY_START, s["ao"], 2)
    return s


def run(s):
    k = s["kind"]
    if k == "frame":
        ep.epbr_ssao(s["gb"], s["cam"], s["ssao"], s["ao"], workspace=s["ws"])
        ep.epbr_shade_tonemap(s["gb"], s["cam"], s["lights"], s["ibl"], s["params"], s["hdr"], s["fmt"], s["tp"], s["ldr"])
        return {"ao": s["ao"], "hdr": s["hdr"], "ldr": s["ldr"]}
    if k == "shadow":
        ep.epbr_shade_shadows(s["gb"], s["cam"], s["lights"], s["ibl"], s["params"], s["shadows"], s["hdr"], s["fmt"],
                              s["tp"], s["ldr"])
    elif k == "maps":
        ep.epbr_shadow_maps(s["mesh"], s["cams"], NEAR, s["maps"], workspace=s["ws"])
        return {"maps": s["maps"]}
    elif k == "mesh":
        ep.epbr_raster_gbuffer(s["mesh"], s["cam"], NEAR, s["gb"], ids=s["ids"], workspace=s["ws"])
        return {"rt0": s["rt"][0], "rt1": s["rt"][1], "depth": s["rt"][2], "ids": s["ids"]}
    elif k == "surfels":
        ep.epbr_surfel_gbuffer(s["surfels"], s["cam"], NEAR, s["case"]["tol"], s["gb"], weight=s["weight"], workspace=s["ws"])
        return {"rt0": s["rt"][0], "rt1": s["rt"][1], "depth": s["rt"][2], "weight": s["weight"]}
    elif k == "bloom":
        ep.epbr_bloom(s["src"], s["fmt"], s["bp"], s["hdr"], s["fmt"], s["tp"], s["ldr"], workspace=s["ws"])
    elif k == "edl":
        ep.epbr_edl(s["gb"], s["ep"], s["hdr"], s["fmt"], tp=s["tp"], ldr=s["ldr"])
    elif k == "ibl":
        ep.epbr_precompute_ibl(s["env"], s["ibl"], workspace=s["ws"])
        ibl = s["ibl"]
        return {"irradiance": ibl.irradiance(), "lut": ibl.lut(),
                "levels": [ibl.level(m) for m in range(s["case"]["levels"])]}
    else:
        s["batch"].launch()
    return {"hdr": s["hdr"], "ldr": s["ldr"]}


# ------------------------------------------------------------------------------------------
# the same outputs in 64 bits, from plain torch
# ------------------------------------------------------------------------------------------
def _dot(a, b):
    return (a * b).sum(-1)


def _rays(sc, W, H):
    t = math.tan(0.5 * sc.fov)
    px = (2.0 * (torch.arange(W, device="cuda", dtype=F64) + 0.5) / W - 1.0) * t * W / H
    py = (1.0 - 2.0 * (torch.arange(H, device="cuda", dtype=F64) + 0.5) / H) * t
    return torch.stack([px[None].expand(H, W), py[:, None].expand(H, W), torch.full((H, W), -1.0, device="cuda", dtype=F64)], 2)


def _view32(sc):
    return _t(sc.view.astype(np.float32), F64)


def _decode(planes):
    """Albedo, metal, unit normal, rough, depth in 64 bits."""
    if len(planes) == 3:
        rt0, rt1, e = (p.double() for p in planes)
        n = rt1[..., :3]
        return rt0[..., :3], rt0[..., 3].clamp(0, 1), n / n.norm(dim=2, keepdim=True), rt1[..., 3].clamp(0.045, 1), e
    c = planes[0][..., :3].double() / 255
    alb = torch.where(c <= 0.04045, c / 12.92, ((c + 0.055) / 1.055) ** 2.4)
    p = planes[1].double()
    z = 1 - p.abs().sum(2)
    fold = (1.0 - p.flip(2).abs()) * torch.where(p >= 0, 1.0, -1.0)
    n = torch.cat([torch.where(z[..., None] < 0, fold, p), z[..., None]], 2)
    mr = planes[2].double() / 255
    return alb, mr[..., 0], n / n.norm(dim=2, keepdim=True), mr[..., 1].clamp(0.045, 1), planes[3].double()


def _basis(n):
    s = torch.where(n[..., 2] >= 0, 1.0, -1.0)
    a = -1.0 / (s + n[..., 2])
    c = n[..., 0] * n[..., 1] * a
    t = torch.stack([1 + s * n[..., 0] ** 2 * a, s * c, -s * n[..., 0]], -1)
    return t, torch.stack([c, s + n[..., 1] ** 2 * a, -n[..., 1]], -1)


def _exact_ssao(sc, planes, kern, noise, W, H, radius=0.5, bias=0.025):
    _, _, n, _, e = _decode(planes)
    R = _view32(sc)[:3, :3]
    P = (e[..., None] * _rays(sc, W, H))[::2, ::2]
    nv = (n @ R)[::2, ::2]
    ea = e[::2, ::2]
    on = torch.isfinite(ea)
    ha, wa = ea.shape
    j, i = torch.meshgrid(torch.arange(ha, device="cuda"), torch.arange(wa, device="cuda"), indexing="ij")
    rv = torch.cat([noise.double()[(j % 4) * 4 + i % 4], torch.zeros(ha, wa, 1, device="cuda", dtype=F64)], 2)
    t = rv - nv * _dot(rv, nv)[..., None]
    tn = t.norm(dim=2, keepdim=True)
    tb, bb = _basis(nv)
    par = tn < 1e-4
    t = torch.where(par, tb, t / tn.clamp_min(1e-9))
    b = torch.where(par, bb, torch.linalg.cross(nv, t, dim=2))
    th = math.tan(0.5 * sc.fov)
    sx, sy = 0.5 * H / th, 0.5 * H / th
    occ = torch.zeros_like(ea)
    for q in kern.double():
        S = P + radius * (t * q[0] + b * q[1] + nv * q[2])
        es = -S[..., 2]
        x, y = torch.floor(S[..., 0] / es * sx + 0.5 * W), torch.floor(-S[..., 1] / es * sy + 0.5 * H)
        ok = on & (es > 0) & (x >= 0) & (y >= 0) & (x < W) & (y < H)
        at = torch.where(ok, y * W + x, 0.0).nan_to_num(0.0).long()
        eb = e.reshape(-1)[at]
        u = (radius / (ea - eb).abs()).clamp(0, 1)
        occ += torch.where(ok & torch.isfinite(eb) & (eb <= es - bias), u * u * (3 - 2 * u), 0.0)
    raw = torch.where(on, 1 - occ / len(kern), 1.0)
    pad = torch.nn.functional.pad
    A, E = pad(raw, (3, 3, 3, 3)), pad(ea, (3, 3, 3, 3), value=INF)
    num, den = torch.zeros_like(ea), torch.zeros_like(ea)
    for dy in range(7):
        for dx in range(7):
            a, q = A[dy:dy + ha, dx:dx + wa], E[dy:dy + ha, dx:dx + wa]
            w = torch.exp(-((dx - 3) ** 2 + (dy - 3) ** 2) / 8.0 - (q - ea).abs() / (0.1 * ea))
            w = torch.where(torch.isfinite(q), w, 0.0)
            num, den = num + w * a, den + w
    return torch.where(on, num / den, 1.0)


def _bilinear(img, x, y, wrap):
    H, W = img.shape[:2]
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = (x - x0)[..., None], (y - y0)[..., None]
    i0, j0 = x0.long(), y0.long()
    i1, j1 = i0 + 1, (j0 + 1).clamp(0, H - 1)
    i0, i1 = (i0 % W, i1 % W) if wrap else (i0.clamp(0, W - 1), i1.clamp(0, W - 1))
    j0 = j0.clamp(0, H - 1)
    f = img.reshape(H * W, -1)
    top = f[j0 * W + i0] * (1 - fx) + f[j0 * W + i1] * fx
    return top * (1 - fy) + (f[j1 * W + i0] * (1 - fx) + f[j1 * W + i1] * fx) * fy


def _lookup(img, d):
    H, W = img.shape[:2]
    u = 0.5 + torch.atan2(d[..., 0], -d[..., 2]) / (2 * math.pi)
    v = torch.atan2((d[..., 0] ** 2 + d[..., 2] ** 2).sqrt(), d[..., 1]) / math.pi
    return _bilinear(img, u * W - 0.5, v * H - 0.5, True)


def _visible(P, cam, m):
    q = P @ cam[:12].view(3, 4)[:, :3].T + cam[:12].view(3, 4)[:, 3]
    z, S = -q[:, 2], m.shape[0]
    s, t = (q[:, 0] * cam[12] / z + 1) * S / 2, (1 - q[:, 1] * cam[12] / z) * S / 2
    i0, j0 = torch.floor(s.clamp(-9, S + 9)).long(), torch.floor(t.clamp(-9, S + 9)).long()
    lit = torch.zeros_like(z)
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            i, j = i0 + dx, j0 + dy
            in_ = (i >= 0) & (j >= 0) & (i < S) & (j < S)
            d = m[j.clamp(0, S - 1), i.clamp(0, S - 1)].double()
            lit += ((~in_) | (z <= d + 0.02 + 0.01 * z)).double()
    return torch.where(z > 0, lit / 9, 1.0)


def _exact_shade(sc, planes, lights, maps, W, H, ao=None, shadow=None):
    lev, irr, lut = [m.double() for m in maps[0]], maps[1].double(), maps[2].double()
    alb, met, n, rough, e = _decode(planes)
    v2w = _view32(sc)
    dw = _rays(sc, W, H) @ v2w[:3, :3].T
    on = torch.isfinite(e).reshape(-1)
    out = torch.empty(H * W, 3, device="cuda", dtype=F64)
    dw = dw.reshape(-1, 3)
    out[~on] = _lookup(lev[0][..., :3], dw[~on])
    alb, n, met, rough, e, dw = (x.reshape(H * W, -1)[on] for x in (alb, n, met, rough, e, dw))
    P = v2w[:3, 3] + e * dw
    v = -dw / dw.norm(dim=1, keepdim=True)
    nvr = _dot(n, v)[:, None]
    nv = nvr.clamp_min(1e-4)
    F0 = 0.04 + met * (alb - 0.04)
    cd = alb * (1 - met)
    a2 = rough ** 4
    k = (rough + 1) ** 2 / 8
    acc = torch.zeros_like(P)
    for i, li in enumerate(lights.double()):
        L = li[:3] - P
        d2 = _dot(L, L)[:, None]
        l = L / d2.sqrt()
        nl = _dot(n, l)[:, None].clamp_min(0)
        s = l + v
        s2 = _dot(s, s)[:, None]
        ns = _dot(n, s)[:, None]
        c = torch.linalg.cross(n, s, dim=1)
        den = ns * ns * a2 + _dot(c, c)[:, None]
        D = a2 * s2 * s2 / (math.pi * den * den)
        G = nl * nv / ((nl * (1 - k) + k) * (nv * (1 - k) + k))
        Fr = F0 + (1 - F0) * (1 - s2.sqrt() / 2) ** 5
        f = (1 - Fr) * cd / math.pi + torch.where(nl > 0, D * G / (4 * nl * nv).clamp_min(1e-300), 0.0) * Fr
        w = nl / d2
        if shadow is not None:
            w = w * _visible(P, shadow[1][i].double(), shadow[0][i])[:, None]
        acc += f * (li[3] * li[4:7]) * w
    ir = _lookup(irr[..., :3], n)
    R = 2 * nvr * n - v
    lod = rough[:, 0] * (len(lev) - 1)
    pref = torch.zeros_like(P)
    for m, img in enumerate(lev):
        w = (1 - (lod - m).abs()).clamp_min(0)
        at = w > 0
        pref[at] += w[at, None] * _lookup(img[..., :3], R[at])
    AB = _bilinear(lut, nvr[:, 0].clamp(1e-4, 1) * 64 - 0.5, rough[:, 0] * 64 - 0.5, False)
    A, B = AB[:, 0:1], AB[:, 1:2]
    kS = F0 + (torch.maximum(1 - rough, F0) - F0) * (1 - nv) ** 5
    Fss = kS * A + B
    Ems = 1 - A - B
    Fa = F0 + (1 - F0) / 21
    Fms = Fss * Fa / (1 - Ems * Fa)
    amb = Fss * pref + (Fms * Ems + cd * (1 - Fss - Fms * Ems)) * ir
    if ao is not None:
        y, x = torch.meshgrid(torch.arange(H, device="cuda") // 2, torch.arange(W, device="cuda") // 2, indexing="ij")
        amb = amb * ao[y, x].reshape(-1)[on][:, None]
    out[on] = acc + amb
    return out.view(H, W, 3)


def _rgba(c):
    return torch.cat([c, torch.ones_like(c[..., :1])], -1)


def _project(verts, view, fov, W, H):
    """Snapped positions and 1/z of every vertex: FP32, each operation rounded, as the pass defines it."""
    t = math.tan(0.5 * float(np.float32(fov)))
    f = np.float32
    kx, ky = float(f(H / (W * t))), float(f(1 / t))
    R, eye = _t(view[:3, :3]), _t(view[:3, 3])
    d = verts[:, :3] - eye
    ax = [(R[0, k] * d[:, 0] + R[1, k] * d[:, 1]) + R[2, k] * d[:, 2] for k in range(3)]
    e = -ax[2]
    iz = 1.0 / e
    X, Y = 0.5 * W * (1.0 + (ax[0] * iz) * kx), 0.5 * H * (1.0 - (ax[1] * iz) * ky)
    ok = (e >= float(f(NEAR))) & (X.abs() < 4194304) & (Y.abs() < 4194304)
    return torch.round(X.where(ok, 0 * X) * 256).long(), torch.round(Y.where(ok, 0 * Y) * 256).long(), iz, ok


def _items(x0, x1, y0, y1, most=1 << 24):
    """Chunks of (index, x, y) over every pixel of the boxes [x0, x1] x [y0, y1]."""
    w, h = (x1 - x0 + 1).clamp_min(0), (y1 - y0 + 1).clamp_min(0)
    cnt = w * h
    ends = cnt.cumsum(0)
    a, total = 0, int(ends[-1]) if len(ends) else 0
    while a < len(cnt) and total:
        base = int(ends[a - 1]) if a else 0
        if base >= total:
            break
        b = max(a + 1, int(torch.searchsorted(ends, base + most)))
        idx = torch.arange(a, min(b, len(cnt)), device="cuda").repeat_interleave(cnt[a:b])
        loc = torch.arange(len(idx), device="cuda") + base - (ends[idx] - cnt[idx])
        yield idx, x0[idx] + loc % w[idx], y0[idx] + loc // w[idx]
        a = b


def _exact_raster(verts, tris, view, fov, W, H):
    """(nearest depth, its triangle, its weights' numerators) of every pixel, -1 where none."""
    qx, qy, iz, ok = _project(verts, view, fov, W, H)
    t = tris.long()
    keep = ok[t].all(1)
    x, y = qx[t], qy[t]
    edge = lambda i, j, px, py, X, Y: (X[:, j] - X[:, i]) * (py - Y[:, i]) - (Y[:, j] - Y[:, i]) * (px - X[:, i])
    area = edge(0, 1, x[:, 2], y[:, 2], x, y)
    flip = (area < 0)[:, None]
    t = torch.where(flip, t[:, [0, 2, 1]], t)
    x, y, area = qx[t], qy[t], area.abs()
    keep &= area > 0
    x0, x1 = ((x.amin(1) + 127) >> 8).clamp_min(0), ((x.amax(1) - 128) >> 8).clamp_max(W - 1)
    y0, y1 = ((y.amin(1) + 127) >> 8).clamp_min(0), ((y.amax(1) - 128) >> 8).clamp_max(H - 1)
    x1 = torch.where(keep, x1, x0 - 1)
    best = torch.full((H * W,), INF, device="cuda", dtype=F64)
    tri = torch.full((H * W,), -1, device="cuda")
    for idx, X, Y in _items(x0, x1, y0, y1):
        xs, ys, px, py = x[idx], y[idx], 256 * X + 128, 256 * Y + 128
        in_ = torch.ones(len(idx), dtype=torch.bool, device="cuda")
        s = torch.zeros(len(idx), device="cuda", dtype=F64)
        for i, j, o in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
            w = edge(i, j, px, py, xs, ys)
            dx, dy = xs[:, j] - xs[:, i], ys[:, j] - ys[:, i]
            in_ &= (w > 0) | ((w == 0) & ((dy < 0) | ((dy == 0) & (dx > 0))))
            s += w.double() * iz[t[idx, o]].double()
        z, p = (area[idx].double() / s)[in_], (Y * W + X)[in_]
        new = torch.full_like(best, INF).scatter_reduce(0, p, z, "amin")
        mine = z == new[p]
        who = torch.full_like(tri, 1 << 40).scatter_reduce(0, p[mine], idx[in_][mine], "amin")
        closer = new < best
        best, tri = torch.where(closer, new, best), torch.where(closer, who, tri)
    return best, tri, t, qx, qy, iz


def _exact_mesh(case, seed):
    W, H = case["width"], case["height"]
    sc = _Scene(seed, case["spheres"])
    verts, tris = _mesh(sc, case["lat"], case["lon"], case["ground"])
    z, tri, t, qx, qy, iz = _exact_raster(verts, tris, sc.view.astype(np.float32), sc.fov, W, H)
    on = tri >= 0
    p = on.nonzero()[:, 0]
    v = t[tri[p]]
    X, Y = 256 * (p % W) + 128, 256 * (p // W) + 128
    x, y = qx[v], qy[v]
    e = lambda i, j: ((x[:, j] - x[:, i]) * (Y - y[:, i]) - (y[:, j] - y[:, i]) * (X - x[:, i])).double()
    w = torch.stack([e(1, 2), e(2, 0), e(0, 1)], 1) * iz[v].double()
    w = w / w.sum(1, keepdim=True)
    at = (w[..., None] * verts.double()[v][:, :, 3:11]).sum(1)
    rt0, rt1 = (torch.zeros(H * W, 4, device="cuda", dtype=F64) for _ in range(2))
    rt0[p] = at[:, 3:7]
    rt1[p] = torch.cat([at[:, :3] / at[:, :3].norm(dim=1, keepdim=True), at[:, 7:]], 1)
    return {"rt0": rt0.view(H, W, 4), "rt1": rt1.view(H, W, 4), "depth": z.view(H, W), "ids": None}


def _exact_surfels(case, seed):
    W, H = case["width"], case["height"]
    sc = _Scene(seed, case["spheres"])
    rec = _surfels(sc, case["per_sphere"], case["ground"], seed)
    f = np.float32
    view = sc.view.astype(np.float32)
    th = math.tan(0.5 * float(f(sc.fov)))
    ky, kx = float(f(1 / th)), float(f(H / (W * th)))
    ax = _t(view[:3, :3])
    dot = lambda a, b: (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2]
    cols = lambda m: [m[:, 0], m[:, 1], m[:, 2]]
    to_view = lambda m: [dot(ax[:, k], cols(m)) for k in range(3)]
    c, n, t = to_view(rec[:, 0:3] - _t(view[:3, 3])), to_view(rec[:, 4:7]), to_view(rec[:, 8:11])
    a, b = rec[:, 3], rec[:, 7]
    inv = 1.0 / dot(n, n).sqrt()
    n = [x * inv for x in n]
    dt = dot(t, n)
    t = [x - y * dt for x, y in zip(t, n)]
    inv = 1.0 / dot(t, t).sqrt()
    t = [x * inv for x in t]
    bt = [n[1] * t[2] - n[2] * t[1], n[2] * t[0] - n[0] * t[2], n[0] * t[1] - n[1] * t[0]]
    ok = (-c[2]) - (a + b) >= float(f(NEAR))
    ia2, ib2 = 1.0 / (a * a), 1.0 / (b * b)
    nc, ct, cb = dot(n, c), dot(c, t), dot(c, bt)
    ux = (((torch.arange(W, device="cuda") + 0.5) / (0.5 * W)) - 1.0) / kx
    uy = (1.0 - (torch.arange(H, device="cuda") + 0.5) / (0.5 * H)) / ky
    # a generous box: the disk's bounding box in view space, projected
    ext = [torch.sqrt((a * t[k]) ** 2 + (b * bt[k]) ** 2).double() for k in range(3)]
    zl, zh = -c[2].double() - ext[2], -c[2].double() + ext[2]
    ok &= zl > 0.5 * NEAR
    def span(k, s, h, lim):
        lo, hi = s * c[k].double() - ext[k], s * c[k].double() + ext[k]
        g = kx if k == 0 else ky
        p0 = h * (1 + g * torch.minimum(lo / zl, lo / zh)) - 0.5
        p1 = h * (1 + g * torch.maximum(hi / zl, hi / zh)) - 0.5
        return (torch.floor(p0) - 1).clamp(0, lim).long(), (torch.ceil(p1) + 1).clamp(-1, lim - 1).long()
    x0, x1 = span(0, 1.0, 0.5 * W, W)
    y0, y1 = span(1, -1.0, 0.5 * H, H)
    x1 = torch.where(ok, x1, x0 - 1)
    depth = torch.full((H * W,), INF, device="cuda")
    acc = torch.zeros(H * W, 9, device="cuda", dtype=F64)
    nw = rec[:, 4:7].double()
    nw = nw / nw.norm(dim=1, keepdim=True)
    mat = torch.cat([rec[:, 12:15], rec[:, 11:12]], 1).double()
    mat = torch.cat([mat, nw, rec[:, 15:16].double(), torch.ones_like(nw[:, :1])], 1)
    win = float(f(1) + f(case["tol"]))
    for step in (0, 1):
        for i, X, Y in _items(x0, x1, y0, y1, 1 << 25):
            u, w = ux[X], uy[Y]
            ray = lambda m: (m[0][i] * u + m[1][i] * w) - m[2][i]
            nd, tt, bb = ray(n), ray(t), ray(bt)
            U, V = nc[i] * tt - nd * ct[i], nc[i] * bb - nd * cb[i]
            hit = (nc[i] * nd > 0) & ((U * U) * ia2[i] + (V * V) * ib2[i] <= nd * nd)
            sd, p, i = (nc[i] / nd)[hit], (Y * W + X)[hit], i[hit]
            if step == 0:
                depth = depth.scatter_reduce(0, p, sd, "amin")
            else:
                in_ = sd <= depth[p] * win
                acc.index_add_(0, p[in_], mat[i[in_]])
    wt = acc[:, 8:9]
    on = wt[:, 0] > 0
    m = torch.where(on[:, None], acc[:, :8] / wt.clamp_min(1), 0.0)
    nn = m[:, 4:7]
    nn = torch.where(on[:, None], nn / nn.norm(dim=1, keepdim=True).clamp_min(1e-30), 0.0)
    return {"rt0": m[:, :4].reshape(H, W, 4), "rt1": torch.cat([nn, m[:, 7:8]], 1).view(H, W, 4),
            "depth": torch.where(on, depth.double(), INF).view(H, W), "weight": wt.view(H, W)}


def _exact_bloom(case, seed):
    W, H = case["width"], case["height"]
    src = _hdr_field(case, seed)[..., :3]
    f = src.float()
    lum = (0.2126 * f[..., 0] + 0.7152 * f[..., 1]) + 0.0722 * f[..., 2]
    src = src.double()
    lev = torch.where((lum > 1.0)[..., None], src, 0.0)
    R, add = case["radius"], torch.zeros_like(src)
    g = torch.exp(-torch.arange(-R, R + 1, device="cuda", dtype=F64) ** 2 / 8.0)
    g = g / g.sum()
    x, y = torch.arange(W, device="cuda", dtype=F64), torch.arange(H, device="cuda", dtype=F64)
    for k in range(1, case["levels"]):
        h, w = lev.shape[:2]
        j = torch.arange((h + 1) // 2, device="cuda") * 2
        i = torch.arange((w + 1) // 2, device="cuda") * 2
        j1, i1 = (j + 1).clamp_max(h - 1), (i + 1).clamp_max(w - 1)
        lev = (lev[j][:, i] + lev[j][:, i1] + lev[j1][:, i] + lev[j1][:, i1]) / 4
        h, w = lev.shape[:2]
        b = sum(g[d + R] * lev[:, (torch.arange(w, device="cuda") + d).clamp(0, w - 1)] for d in range(-R, R + 1))
        b = sum(g[d + R] * b[(torch.arange(h, device="cuda") + d).clamp(0, h - 1)] for d in range(-R, R + 1))
        X, Y = torch.meshgrid((x + 0.5) / 2 ** k - 0.5, (y + 0.5) / 2 ** k - 0.5, indexing="xy")
        add += _bilinear(b, X, Y, False)
    return {"hdr": _rgba(src + 0.5 * add), "ldr": None}


def _exact_edl(case, seed):
    planes = _cloud(case, seed)
    e = planes[-1].double()
    H, W = e.shape
    if case["compact"]:
        c = planes[0][..., :3].double() / 255
        c = torch.where(c <= 0.04045, c / 12.92, ((c + 0.055) / 1.055) ** 2.4)
    else:
        c = planes[0][..., :3].double()
    R, N = case["radius"], case["directions"]
    l = torch.nn.functional.pad(torch.log2(e), (R, R, R, R), value=INF)
    on = torch.isfinite(e)
    w = torch.zeros_like(e)
    half = lambda v: int(math.copysign(math.floor(abs(v) + 0.5), v))
    for k in range(N):
        a = 2 * math.pi * k / N
        dx, dy = half(round(R * math.cos(a), 9)), half(round(R * math.sin(a), 9))
        q = l[R + dy:R + dy + H, R + dx:R + dx + W]
        w += torch.where(on & torch.isfinite(q), torch.log2(e) - q, 0.0).clamp_min(0)
    return {"hdr": _rgba(torch.where(on[..., None], c * torch.exp(-8.0 * w / N)[..., None], 0.0)), "ldr": None}


def _sphere_dirs(W, H):
    phi = 2 * math.pi * ((torch.arange(W, device="cuda", dtype=F64) + 0.5) / W - 0.5)
    th = math.pi * (torch.arange(H, device="cuda", dtype=F64) + 0.5) / H
    return torch.stack([th.sin()[:, None] * phi.sin(), th.cos()[:, None].expand(H, W), -th.sin()[:, None] * phi.cos()], 2)


def _ggx(N, a2):
    """Tangent-space half vectors of N Hammersley points; a2 may be a column of values."""
    k = torch.arange(N, device="cuda")
    bits, x2 = k.clone(), torch.zeros(N, device="cuda", dtype=F64)
    for q in range(24):
        x2 += ((bits >> q) & 1).double() * 2.0 ** -(q + 1)
    c2 = (1 - x2) / (1 + (a2 - 1) * x2)
    st, phi = (1 - c2).clamp_min(0).sqrt(), 2 * math.pi * k.double() / N
    return st * phi.cos(), st * phi.sin(), c2.sqrt()


def _exact_ibl(case, seed):
    We, He, M = case["env_w"], case["env_h"], case["levels"]
    env = _sky(seed, We, He).double()
    S, N = case["lut"], case["lut_samples"]
    x = (torch.arange(S, device="cuda", dtype=F64) + 0.5) / S
    lut = torch.zeros(S, S, 2, device="cuda", dtype=F64)
    for j in range(S):
        al = float(x[j]) ** 2
        hx, hy, hz = _ggx(N, al * al)
        mu = x[:, None]
        vh = (1 - mu * mu).sqrt() * hx + mu * hz
        nl = 2 * vh * hz - mu
        k = al / 2
        G = nl / (nl * (1 - k) + k) * mu / (mu * (1 - k) + k) * vh / (hz * mu)
        fc = (1 - vh) ** 5
        G = torch.where(nl > 0, G, 0.0)
        lut[j] = torch.stack([((1 - fc) * G).sum(1), (fc * G).sum(1)], 1) / N
    d = _sphere_dirs(We, He)
    row = math.pi * torch.arange(He + 1, device="cuda", dtype=F64) / He
    om = (2 * math.pi / We) * (row[:-1].cos() - row[1:].cos())
    n = _sphere_dirs(32, 16).reshape(-1, 3)
    num = torch.zeros(512, 4, device="cuda", dtype=F64)
    L = _rgba(env[..., :3])
    for j in range(0, He, 16):
        w = (n @ d[j:j + 16].reshape(-1, 3).T).clamp_min(0)
        num += w @ (L[j:j + 16] * om[j:j + 16, None, None]).reshape(-1, 4)
    levels = [env]
    for m in range(1, M):
        W, H = max(1, We >> m), max(1, He >> m)
        hx, hy, hz = _ggx(case["samples"], (m / (M - 1)) ** 4)
        lx, ly, lz = 2 * hz * hx, 2 * hz * hy, 2 * hz * hz - 1
        keep = lz > 0
        lx, ly, lz = lx[keep], ly[keep], lz[keep]
        nd = _sphere_dirs(W, H).reshape(-1, 3)
        T = torch.linalg.cross(torch.tensor([[0.0, 1.0, 0.0]], device="cuda", dtype=F64).expand_as(nd), nd, dim=1)
        T = T / T.norm(dim=1, keepdim=True)
        B = torch.linalg.cross(nd, T, dim=1)
        out = torch.zeros(W * H, 3, device="cuda", dtype=F64)
        step = max(1, (1 << 24) // (W * H))
        for q in range(0, len(lz), step):
            a, b, c = (v[q:q + step, None, None] for v in (lx, ly, lz))
            out += (_lookup(env[..., :3], T * a + B * b + nd * c) * c).sum(0)
        levels.append(_rgba((out / lz.sum()).view(H, W, 3)))
    return {"irradiance": _rgba(num[:, :3] / num[:, 3:]).view(16, 32, 4), "lut": lut, "levels": levels}


def exact(case, seed):
    k = case["kind"]
    if k == "ibl":
        return _exact_ibl(case, seed)
    if k == "mesh":
        return _exact_mesh(case, seed)
    if k == "surfels":
        return _exact_surfels(case, seed)
    if k == "bloom":
        return _exact_bloom(case, seed)
    if k == "edl":
        return _exact_edl(case, seed)
    if k == "maps":
        sc = _Scene(seed, case["spheres"], case["lights"])
        verts, tris = _mesh(sc, case["lat"], case["lon"], case["ground"])
        S = case["size"]
        return {"maps": torch.stack([_exact_raster(verts, tris, v.astype(np.float32), math.radians(90.0), S, S)[0].view(S, S)
                                     for v in _light_cameras(sc)])}
    W, H = case["width"], case["height"]
    if k == "batch":
        kern, noise = _ssao_inputs(seed, case["samples"])
        maps = [_maps_of(seed + e, case["env"], case["levels"]) for e in range(2)]
        hdr = []
        for v, nl in enumerate(_batch_lights(case, seed)):
            sc = _Scene(seed * 1000 + v, case["spheres"], nl)
            planes = _planes(sc, W, H, False)
            ao = _exact_ssao(sc, planes, kern, noise, W, H)
            hdr.append(_rgba(_exact_shade(sc, planes, _t(sc.lights), maps[v % 2], W, H, ao)))
        return {"hdr": torch.stack(hdr), "ldr": None}
    sc = _Scene(seed, case["spheres"], case["lights"], case["colour"])
    planes = _planes(sc, W, H, bool(case.get("compact")))
    maps = _maps_of(seed, case.get("env", 1024), case.get("levels", 8))
    if k == "shadow":
        sh = _shadow_inputs(sc, case["size"])
        return {"hdr": _rgba(_exact_shade(sc, planes, _t(sc.lights), maps, W, H, None, sh)), "ldr": None}
    kern, noise = _ssao_inputs(seed, case["samples"])
    ao = _exact_ssao(sc, planes, kern, noise, W, H)
    return {"ao": ao, "hdr": _rgba(_exact_shade(sc, planes, _t(sc.lights), maps, W, H, ao)), "ldr": None}

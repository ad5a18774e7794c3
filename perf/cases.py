"""What a user of this renderer has it do, as cases that can be timed and checked.

A case is one call sequence of the package's public entry points on a light field,
an image batch or a refiner; its sizes come from the repository's own configurations
(the tiny cap rig, the full-sphere rig, the eye batch, the two-level loop, the
prefilter, the refinement and its training) and from the ranges around them:
  render    light field -> eye images: plain, without allocations, refined, or
            delivered to host memory
  batch     many eyes of mixed sizes in one call
  levels    the progressive loop: draw what is resident, ask, stream pages
  prefilter source images re-derived from a denser model
  refine    the learned refinement of finished images
  train     training steps of the refinement on image pairs

The light fields are analytic (textured spheres inside a backdrop sphere), ray cast
here with torch.  exact() restates each path in 64 bits with torch alone.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

import paper_1810_08860_gb300 as lfm
from paper_1810_08860_gb300 import disks

RADIUS = 0.35     # capture sphere, metres
Z_NEAR = 0.1
TEX = ("f32", "u8", "bf16", "fp8")
TEX_BYTES = {"f32": 16, "u8": 4, "bf16": 8, "fp8": 4}
BATCH_SIZES = ((512, 512), (1024, 1024), (1440, 1600), (2048, 2048))
TRAIN_LR = 1e-3
TRAIN_SETS = 2    # batches a training pass goes through


def _render(name, **kw):
    c = dict(name=name, kind="render", form="plain", rig="sphere", views=256, size=512, grid=64, tex="f32", mesh="f32",
             disk="round", eyes=2, eye_w=1440, eye_h=1600, spheres=24)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest frame: the repository's tiny cap rig and one 256^2 eye, the preview window of a
        # viewer.  Launches and the host's share count.
        _render("tiny_eye", rig="cap", views=16, size=128, grid=32, eyes=1, eye_w=256, eye_h=256, spheres=8),
        # A plug-in with a frame deadline that may not allocate: the no-allocation entry point close to its
        # limits (32 views, 33^2 meshes), u8 storage, an eye whose sides no tile divides.
        _render("static_u8", form="static", rig="cap", views=30, size=256, grid=33, tex="u8", eyes=1, eye_w=731,
                eye_h=517, spheres=8),
        # The headline: a headset frame from the full 1,024-view rig.
        _render("rig_stereo", views=1024, size=1024),
        # The storage a deployment that must save memory picks (half-size textures, FP16 meshes), on a rig
        # of half the views and a window of odd size.
        _render("ragged_bf16", views=512, tex="bf16", mesh="f16", eye_w=1081, eye_h=1203),
        # Oval disks and the smallest texels, one wide mono window.
        _render("oval_fp8", views=256, tex="fp8", mesh="f16", disk="oval", eyes=1, eye_w=1921, eye_h=1083),
        # The refined frame, read back: what an encoder or a remote client asks for, three frames in flight.
        _render("host_refined", form="host", views=256, size=512, eye_w=1440, eye_h=1600),
        # Offline rendering of many poses: the repository's batch (mixed sizes, cap rig) with 64 eyes.
        dict(name="batch_64", kind="batch", views=16, size=128, grid=32, tex="f32", eyes=64, spheres=8),
        # Two-level progressive frames: a stereo frame from whatever is resident, then the pages it asked for.
        dict(name="levels", kind="levels", fine=512, coarse=128, size=512, grid=64, pages=160, budget=8, eye_w=1440,
             eye_h=1600, spheres=24),
        # Prefiltering a block of source images from a model with 4 times the views and 256^2 meshes.
        dict(name="prefilter", kind="prefilter", views=64, size=512, grid=64, dense=256, dense_grid=256, samples=32,
             block=2, spheres=24),
        # The refinement of a finished stereo frame by the fused kernel, and the default per-layer one on a
        # small odd image.
        dict(name="refine_stereo", kind="refine", kernel="fused", n=2, h=1600, w=1440),
        dict(name="refine_window", kind="refine", kernel="layers", n=1, h=517, w=731),
        # Training at the repository's batch (16 crops of 256^2), the state read back as for a checkpoint.
        dict(name="train_16x256", kind="train", n=16, h=256, w=256, steps=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "batch", "levels", "prefilter", "refine", "refine", "train"])
    if kind == "render":
        form = rng.choice(["plain", "plain", "static", "host", "refined"])
        if form == "static":
            return {k: v for k, v in _render("", form=form, rig="cap", views=rng.randint(4, 32), size=_log(rng, 64, 512),
                                             grid=rng.randint(9, 33), tex=rng.choice(TEX), mesh=rng.choice(("f32", "f16")),
                                             disk="round", eyes=1, eye_w=_log(rng, 96, 1024), eye_h=_log(rng, 96, 1024),
                                             spheres=8).items() if k != "name"}
        return {k: v for k, v in _render("", form=form, views=_log(rng, 48, 512), size=_log(rng, 96, 512),
                                         grid=_log(rng, 16, 129), tex=rng.choice(TEX), mesh=rng.choice(("f32", "f16")),
                                         disk=rng.choice(("round", "round", "oval")), eyes=rng.randint(1, 2),
                                         eye_w=_log(rng, 96, 1600), eye_h=_log(rng, 96, 1600)).items() if k != "name"}
    if kind == "batch":
        return dict(kind=kind, views=rng.choice((9, 16, 25)), size=_log(rng, 96, 512), grid=rng.randint(16, 64),
                    tex=rng.choice(TEX), eyes=rng.randint(3, 48), spheres=rng.randint(4, 16))
    if kind == "levels":
        fine = _log(rng, 96, 512)
        return dict(kind=kind, fine=fine, coarse=fine // 4, size=_log(rng, 96, 512), grid=_log(rng, 17, 65),
                    pages=rng.randint(fine // 5, fine // 2), budget=rng.randint(2, 12), eye_w=_log(rng, 200, 1500),
                    eye_h=_log(rng, 200, 1500), spheres=24)
    if kind == "prefilter":
        return dict(kind=kind, views=rng.randint(40, 80), size=_log(rng, 96, 512), grid=_log(rng, 17, 65),
                    dense=rng.randint(150, 256), dense_grid=_log(rng, 65, 257), samples=rng.randint(9, 32), block=rng.randint(1, 2),
                    spheres=24)
    if kind == "refine":
        return dict(kind=kind, kernel=rng.choice(("fused", "layers")), n=rng.randint(1, 2), h=_log(rng, 64, 1600),
                    w=_log(rng, 64, 1440))
    return dict(kind="train", n=rng.randint(1, 16), h=rng.randint(64, 256), w=rng.randint(64, 256), steps=rng.randint(2, 8))


# ------------------------------------------------------------------ light fields


def _look(forward):
    z = np.asarray(forward, float) / np.linalg.norm(forward)
    d = np.array([0.0, 1.0, 0.0]) if abs(z[1]) < 0.999 else np.array([0.0, 0.0, 1.0])
    y = d - (d @ z) * z
    y /= np.linalg.norm(y)
    return np.stack([np.cross(y, z), y, z], axis=1)


def _pose(R, t):
    return np.concatenate([np.asarray(R, float).reshape(9), np.asarray(t, float)])


def _intr(w, h, hfov):
    f = 0.5 * w / math.tan(0.5 * math.radians(hfov))
    return np.array([f, f, 0.5 * w, 0.5 * h])


def _yaw_pitch(yaw, pitch):
    return np.array([math.cos(pitch) * math.sin(yaw), -math.sin(pitch), math.cos(pitch) * math.cos(yaw)])


def _sphere_dirs(n):
    k = np.arange(n)
    z = 1.0 - (2.0 * k + 1.0) / n
    s, phi = np.sqrt(1.0 - z * z), k * math.pi * (3.0 - math.sqrt(5.0))
    return np.stack([s * np.cos(phi), s * np.sin(phi), z], axis=1)


def _cap_dirs(n, cap_deg=40.0):
    rows = math.isqrt(n - 1) + 1
    cols = -(-n // rows)
    a = np.radians(np.linspace(-cap_deg / 2, cap_deg / 2, max(2, rows)))
    b = np.radians(np.linspace(-cap_deg / 2, cap_deg / 2, max(2, cols)))
    return np.stack([_yaw_pitch(y, p) for p in a for y in b])[:n]


def _scene(rng, n_spheres, cone_deg=None):
    """Spheres (centre, radius, two colours, checker period), then the backdrop (radius 6 m)."""
    out = []
    for _ in range(n_spheres):
        if cone_deg is None:
            d = rng.normal(size=3)
        else:
            cz, phi = rng.uniform(math.cos(math.radians(cone_deg)), 1.0), rng.uniform(0.0, 2.0 * math.pi)
            d = np.array([math.sqrt(1 - cz * cz) * math.cos(phi), math.sqrt(1 - cz * cz) * math.sin(phi), cz])
        c = d / np.linalg.norm(d) * rng.uniform(1.5, 4.0)
        out.append((c, rng.uniform(0.2, 0.6), rng.uniform(0.15, 0.95, 3), rng.uniform(0.05, 0.6, 3), rng.uniform(0.08, 0.25)))
    out.append((np.zeros(3), 6.0, rng.uniform(0.5, 0.9, 3), rng.uniform(0.1, 0.4, 3), 0.6))
    return out


def _cast(scene, o, d):
    """Nearest hit of rays o + t d (d: 3 planes of one shape, not normalised): t and the object's index."""
    best = torch.full_like(d[0], float("inf"))
    which = torch.zeros(d[0].shape, dtype=torch.int64, device=best.device)
    qa = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    for k, (c, r, _, _, _) in enumerate(scene):
        oc = [o[i] - float(c[i]) for i in range(3)]
        qb = d[0] * oc[0] + d[1] * oc[1] + d[2] * oc[2]
        qc = oc[0] * oc[0] + oc[1] * oc[1] + oc[2] * oc[2] - r * r
        s = torch.sqrt(torch.clamp(qb * qb - qa * qc, min=0.0))
        t = (-qb + (s if k == len(scene) - 1 else -s)) / qa
        hit = (qb * qb > qa * qc) & (t > 1e-6) & (t < best)
        best = torch.where(hit, t, best)
        which = torch.where(hit, k, which)
    return best, which


def _rays(poses, intr, u, v):
    """Origins and directions (z component 1 in the camera) of image points u, v (broadcast) of n cameras."""
    R, t = poses[:, :9].reshape(-1, 3, 3), poses[:, 9:]
    x, y = (u - intr[0]) / intr[1], (v - intr[2]) / intr[3]
    sh = (-1,) + (1,) * x.dim()
    d = [R[:, k, 0].reshape(sh) * x + R[:, k, 1].reshape(sh) * y + R[:, k, 2].reshape(sh) for k in range(3)]
    return [t[:, k].reshape(sh).expand_as(d[k]) for k in range(3)], d


def _light_field(scene, dirs, size, grid, hfov, disk_scale=1.2):
    dev = "cuda"
    n = len(dirs)
    poses = np.stack([_pose(_look(d), RADIUS * d) for d in dirs])
    K = _intr(size, size, hfov)
    k = (float(K[2]), float(K[0]), float(K[3]), float(K[1]))
    colours = torch.tensor(np.stack([np.stack([s[2], s[3]]) for s in scene]), dtype=torch.float32, device=dev)
    periods = torch.tensor([s[4] for s in scene], dtype=torch.float32, device=dev)
    centres = torch.tensor(np.stack([s[0] for s in scene]), dtype=torch.float32, device=dev)
    images = np.empty((n, size, size, 4), np.uint8)
    px = torch.arange(size, device=dev, dtype=torch.float32) + 0.5
    chunk = max(1, (1 << 24) // (size * size))
    P32 = torch.tensor(poses, dtype=torch.float32, device=dev)
    for a in range(0, n, chunk):
        o, d = _rays(P32[a:a + chunk], k, px[None, :].expand(size, size), px[:, None].expand(size, size))
        t, w = _cast(scene, o, d)
        per, cen = periods[w], centres[w]
        cell, wave = None, None
        for i in range(3):
            q = (o[i] + t * d[i] - cen[..., i]) / per
            f = torch.floor(q).to(torch.int32)
            cell = f if cell is None else cell + f
            s = torch.sin(q * (2.3 + i))
            wave = s if wave is None else wave * s
        rgb = torch.where((cell & 1).bool()[..., None], colours[w, 0], colours[w, 1]) * (0.8 + 0.2 * wave[..., None])
        out = torch.full(rgb.shape[:-1] + (4,), 255, dtype=torch.uint8, device=dev)
        out[..., :3] = (rgb.clamp(0.0, 1.0) * 255.0 + 0.5).to(torch.uint8)
        torch.from_numpy(images[a:a + chunk]).copy_(out)
        del o, d, t, w, per, cen, cell, wave, rgb, out
    e = torch.arange(grid, device=dev, dtype=torch.float64) * (size / (grid - 1))
    depth = np.empty((n, grid, grid), np.float32)
    P64 = torch.tensor(poses, device=dev)
    for a in range(0, n, 64):
        o, d = _rays(P64[a:a + 64], k, e[None, :].expand(grid, grid), e[:, None].expand(grid, grid))
        depth[a:a + 64] = _cast(scene, o, d)[0].to(torch.float32).cpu().numpy()
    c = RADIUS * np.asarray(dirs)
    nn = torch.cdist(torch.tensor(c, device=dev), torch.tensor(c, device=dev)) + 10.0 * torch.eye(n, device=dev, dtype=torch.float64)
    r = disk_scale * float(nn.amin(1).mean())
    return SimpleNamespace(poses=poses, intr=np.tile(K, (n, 1)), width=size, height=size, images=images, grid_n=grid,
                           depth=depth, disk_c=c.astype(np.float32), disk_r=np.full(n, r, np.float32), sphere_c=np.zeros(3),
                           sphere_r=RADIUS, disk_ext=None)


def _case_light_field(c, rng):
    if c.get("rig", "cap") == "cap":
        scene = _scene(rng, c["spheres"], cone_deg=35.0)
        lf = _light_field(scene, _cap_dirs(c["views"]), c["size"], c["grid"], 90.0)
    else:
        scene = _scene(rng, c["spheres"])
        lf = _light_field(scene, _sphere_dirs(c["views"]), c["size"], c["grid"], 120.0)
    if c.get("disk") == "oval":
        lf.disk_ext = disks.oval_extents(lf)
    return lf


def _head(rng, w, h, eyes, cap):
    """A head inside the rig: the cap rig is looked at along its axis, the full sphere anywhere within
    +-60 degrees of the horizon; a stereo pair stands 64 mm apart."""
    while True:
        centre = rng.uniform(-0.2, 0.2, 3)
        if centre @ centre <= 0.04:
            break
    lim = math.radians(10.0)
    yaw, pitch = (rng.uniform(-lim, lim, 2) if cap else (rng.uniform(0, 2 * math.pi), rng.uniform(-1.0, 1.0) * math.pi / 3))
    return _eyes(centre, yaw, pitch, w, h, eyes, 90.0 if cap else 100.0)


def _eyes(centre, yaw, pitch, w, h, eyes, hfov):
    R = _look(_yaw_pitch(yaw, pitch))
    K = _intr(w, h, hfov)
    off = [0.0] if eyes == 1 else [-0.032, 0.032]
    return [SimpleNamespace(pose=_pose(R, centre + o * R[:, 0]), intr=K, width=w, height=h) for o in off]


def _images(rng, n, h, w):
    """Finished renders: smooth colour fields with edges, 2 % of the pixels empty."""
    dev = "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(rng.integers(1 << 62)))
    y = torch.arange(h, device=dev, dtype=torch.float32)[:, None]
    x = torch.arange(w, device=dev, dtype=torch.float32)[None, :]
    f = rng.uniform(0.02, 0.3, (n, 3, 2))
    rgb = torch.stack([torch.stack([0.5 + 0.3 * torch.sin(float(f[i, k, 0]) * x + float(f[i, k, 1]) * y)
                                    + 0.1 * torch.sign(torch.sin(0.11 * (k + 1) * x + 0.07 * y)) for k in range(3)], -1)
                       for i in range(n)])
    alpha = (torch.rand((n, h, w, 1), device=dev, generator=gen) > 0.02).to(torch.float32)
    return torch.cat([rgb.clamp(0.0, 1.0) * alpha, alpha], -1).contiguous()


# ------------------------------------------------------------------ the cases' states


def _make(c, seed):
    """Everything the seed decides, before anything is loaded."""
    rng = np.random.default_rng([seed, 1810])
    s = SimpleNamespace(kind=c["kind"], case=c)
    if c["kind"] == "render":
        s.lf = _case_light_field(c, rng)
        s.heads = [_head(rng, c["eye_w"], c["eye_h"], c["eyes"], c["rig"] == "cap") for _ in range(3 if c["form"] == "host" else 1)]
        s.params = _weights(rng)
    elif c["kind"] == "batch":
        s.lf = _case_light_field(c, rng)
        s.eyes = []
        sizes = rng.permutation(np.resize(np.arange(len(BATCH_SIZES)), (c["eyes"] + 1) // 2))
        for k in sizes:
            s.eyes += _head(rng, *BATCH_SIZES[k], 2, True)
        s.eyes = s.eyes[:c["eyes"]]
    elif c["kind"] == "levels":
        scene = _scene(rng, c["spheres"])
        fine = _light_field(scene, _sphere_dirs(c["fine"]), c["size"], c["grid"], 120.0)
        coarse = _light_field(scene, _sphere_dirs(c["coarse"]), c["size"], c["grid"], 120.0)
        for key in ("poses", "intr", "images", "depth", "disk_c", "disk_r"):
            setattr(fine, key, np.concatenate([getattr(fine, key), getattr(coarse, key)]))
        s.lf = fine
        s.centre, s.yaw = rng.uniform(-0.1, 0.1, 3), rng.uniform(0.0, 2.0 * math.pi)
        s.first = rng.permutation(c["fine"])[:c["pages"]]
    elif c["kind"] == "prefilter":
        scene = _scene(rng, c["spheres"])
        s.lf = _light_field(scene, _sphere_dirs(c["views"]), c["size"], c["grid"], 120.0)
        s.dense = _light_field(scene, _sphere_dirs(c["dense"]), c["size"], c["dense_grid"], 120.0)
        s.view = int(rng.integers(0, c["views"] - c["block"] + 1))
        s.samples = _balanced_samples(c["samples"], int(rng.integers(1 << 30)))
    elif c["kind"] == "refine":
        s.params = _weights(rng)
        s.images = _images(rng, c["n"], c["h"], c["w"])
    else:
        s.params = lfm.init_refiner_params(int(rng.integers(1 << 30)))
        s.pairs = []
        for _ in range(TRAIN_SETS):
            x = _images(rng, c["n"], c["h"], c["w"])
            t = x.clone()
            ramp = 0.05 * torch.sin(0.05 * torch.arange(c["w"], device=x.device, dtype=torch.float32))
            t[..., :3] = (x[..., :3] * 0.9 + ramp[None, None, :, None]).clamp(0.0, 1.0) * x[..., 3:]
            s.pairs.append((x, t))
    return s


def _weights(rng):
    """Refiner weights of the size that training leaves: He-normal layers, small biases, a small last layer."""
    p = lfm.init_refiner_params(int(rng.integers(1 << 30)))
    for a, b in ((864, 896), (10112, 10144), (11008, 11011)):
        p[a:b] = rng.normal(0.0, 0.02, b - a)
    return p


def _balanced_samples(n, seed):
    """A sample set whose Lanczos lobes do not nearly cancel, chosen as the benchmark chooses it."""
    while True:
        S = lfm.prefilter_samples(n, seed)
        w = _sample_weights(S)
        if w.sum() > 0.6 * np.abs(w).sum():
            return S
        seed += 1


def _sample_weights(S):
    S = S.astype(np.float64)
    return (1.0 - np.sqrt(S[:, 0])) * np.sinc(S[:, 2]) * np.sinc(S[:, 2] / 2) * np.sinc(S[:, 3]) * np.sinc(S[:, 3] / 2)


def _level_eyes(s, frame):
    c = s.case
    return _eyes(s.centre, s.yaw + math.radians(0.6) * frame, 0.0, c["eye_w"], c["eye_h"], 2, 100.0)


def prepare(case, seed):
    c = case
    s = _make(c, seed)
    if s.kind in ("render", "batch", "levels"):
        eyes = {"render": lambda: s.heads[0], "batch": lambda: s.eyes, "levels": lambda: _level_eyes(s, 0)}[s.kind]()
        s.r = lfm.Renderer(0, max_eyes=max(2, len(eyes)))
        s.r.load_views(s.lf, tex_format=c.get("tex", "f32"))
        s.r.build_meshes(s.lf, mesh_format=c.get("mesh", "f32"))
    if s.kind == "render":
        if c["form"] in ("host", "refined"):
            s.r.load_refiner(s.params)
            s.r.set_refine_kernel("fused")
        if c["form"] == "host":
            s.out = [[torch.empty((e.height, e.width, 4), pin_memory=True) for e in head] for head in s.heads]
        else:
            s.out = [torch.empty((e.height, e.width, 4), device="cuda") for e in s.heads[0]]
        del s.lf
    elif s.kind == "batch":
        s.flat = torch.empty((sum(e.height * e.width for e in s.eyes), 4), device="cuda")
        at = np.cumsum([0] + [e.height * e.width for e in s.eyes])
        s.out = [s.flat[a:b].view(e.height, e.width, 4) for e, a, b in zip(s.eyes, at, at[1:])]
        del s.lf
    elif s.kind == "levels":
        s.r.set_levels(c["fine"], c["pages"])
        s.host = torch.from_numpy(s.lf.images[:c["fine"]]).pin_memory().numpy()
        s.cache = lfm.PageCache(c["fine"], c["pages"])
        _stream_pages(s, s.cache.frame(s.first, c["pages"]))
        s.frame = 0
        s.out = [torch.empty((c["eye_h"], c["eye_w"], 4), device="cuda") for _ in range(2)]
        del s.lf
    elif s.kind == "prefilter":
        s.r = lfm.Renderer(0)
        s.r.load_views(s.lf)
        s.r.build_meshes(s.lf)
        s.rd = lfm.Renderer(0, max_eyes=c["samples"], tri_capacity=c["samples"] << 20)
        s.rd.load_views(s.dense, tex_format="u8")
        s.rd.build_meshes(s.dense)
        s.out = torch.empty((c["block"], c["size"], c["size"], 4), device="cuda")
        del s.lf, s.dense
    else:
        s.r = lfm.Renderer(0)
        s.r.load_refiner(s.params)
        if s.kind == "refine":
            s.r.set_refine_kernel(c["kernel"])
            s.out = torch.empty_like(s.images)
    return s


def _stream_pages(s, admitted):
    if admitted:
        s.r.upload_pages([v for v, _ in admitted], [p for _, p in admitted], [s.host[v] for v, _ in admitted])


def run(state):
    s = state
    c = s.case
    if s.kind == "render":
        if c["form"] == "static":
            return s.r.render_static(s.heads[0][0], out=s.out[0])
        if c["form"] == "refined":
            return s.r.render_refined(s.heads[0], out=s.out)
        if c["form"] == "host":
            for head, out in zip(s.heads, s.out):
                frame, _ = s.r.render_host(head, out=out, form="refined")
            s.r.host_wait(frame)
            return s.out
        return s.r.render(s.heads[0], out=s.out)
    if s.kind == "batch":
        s.r.render_batch(s.eyes, out=s.out)
        return s.flat
    if s.kind == "levels":
        s.r.render(_level_eyes(s, s.frame), out=s.out)
        s.frame += 1
        wanted = s.r.levels_wanted()
        _stream_pages(s, s.cache.frame(wanted, c["budget"]))
        seen = np.zeros(c["fine"], np.uint8)
        seen[wanted] = 1
        return {"images": s.out, "wanted": seen, "pages": s.cache.pages()}
    if s.kind == "prefilter":
        return s.r.prefilter(s.rd, s.samples, first_view=s.view, n_views=c["block"], out=s.out)
    if s.kind == "refine":
        return s.r.refine(s.images, out=s.out)
    for k in range(c["steps"]):
        x, t = s.pairs[k % len(s.pairs)]
        s.r.refine_train_step(x, t, TRAIN_LR)
    return s.r.get_refiner()


def work(case):
    """Bytes: source texels that the frame's pixels see (about four views a pixel; a stereo pair shares
    them), the meshes of the views in sight, and the images written.  Operations: the network's."""
    c = case
    if c["kind"] in ("refine", "train"):
        px = c["n"] * c["h"] * c["w"]
        if c["kind"] == "refine":
            return {"bytes": 32 * px, "flops": 21312 * px}
        return {"bytes": 32 * px * c["steps"] + 16 * lfm.REFINE_N_PARAMS, "flops": 63936 * px * c["steps"]}

    def frame(px_eye, n_out, f_eye, f_src, size, n_views, grid, tb, mb, in_sight):
        seen = px_eye * 4.1 * min(1.0, (f_src / f_eye) ** 2)
        return min(seen, n_views * size * size) * tb + in_sight * n_views * grid * grid * mb + 16 * n_out

    if c["kind"] == "batch":
        eyes = [BATCH_SIZES[k] for k in np.resize(np.arange(len(BATCH_SIZES)), (c["eyes"] + 1) // 2)]
        px = sum(2 * w * h for w, h in eyes) * c["eyes"] // (2 * len(eyes))
        return {"bytes": c["views"] * (c["size"] ** 2 * TEX_BYTES[c["tex"]] + c["grid"] ** 2 * 4) + 16 * px, "flops": 0}
    if c["kind"] == "levels":
        f, g = _intr(c["eye_w"], c["eye_h"], 100.0)[0], _intr(c["size"], c["size"], 120.0)[0]
        px = c["eye_w"] * c["eye_h"]
        return {"bytes": frame(px, 2 * px, f, g, c["size"], c["fine"], c["grid"], 16, 4, 0.5)
                + c["budget"] * c["size"] ** 2 * 20, "flops": 0}
    if c["kind"] == "prefilter":
        px = c["size"] ** 2
        per_view = min(c["dense"], 12) * (px * 4 + c["dense_grid"] ** 2 * 4) + px * 16 + c["grid"] ** 2 * 4
        return {"bytes": c["block"] * per_view, "flops": 0}
    cap = c["rig"] == "cap"
    f, g = _intr(c["eye_w"], c["eye_h"], 90.0 if cap else 100.0)[0], _intr(c["size"], c["size"], 90.0 if cap else 120.0)[0]
    px, frames = c["eye_w"] * c["eye_h"], 3 if c["form"] == "host" else 1
    one = frame(px, c["eyes"] * px, f, g, c["size"], c["views"], c["grid"], TEX_BYTES[c["tex"]], 4 if c["mesh"] == "f32" else 2,
                1.0 if cap else 0.5)
    return {"bytes": frames * one, "flops": 21312 * frames * c["eyes"] * px if c["form"] in ("host", "refined") else 0}


# ------------------------------------------------------------------ the same in 64 bits


def _stored(lf, tex="f32", mesh="f32"):
    """The light field as its storage formats define it, on the device: texel planes per view (a function)
    and 64-bit depths."""
    depth = torch.tensor(lf.depth, device="cuda")
    if mesh == "f16":
        z0 = depth.amin((1, 2), keepdim=True)
        depth = z0 + (depth - z0).to(torch.float16).to(torch.float32)

    def texels(v):
        rgb = torch.from_numpy(lf.images[v])[..., :3].cuda().to(torch.float64)
        if tex == "bf16":
            return (rgb / 255.0).to(torch.bfloat16).to(torch.float64)
        if tex == "fp8":
            scale = rgb.max() / 255.0 / 448.0
            return (rgb / 255.0 / scale).to(torch.float32).to(torch.float8_e4m3fn).to(torch.float64) * scale
        return rgb / 255.0

    return SimpleNamespace(lf=lf, depth=depth.to(torch.float64), texels=texels, cache={})


def _disk_rho(lf, v, d, o, p, ok):
    """Inside the disk of view v?, and its weight there, for rays o + t d with sphere crossings p."""
    c = torch.tensor(lf.disk_c[v].astype(np.float64), device="cuda")
    if lf.disk_ext is None:
        dist2 = (p[0] - c[0]) ** 2 + (p[1] - c[1]) ** 2 + (p[2] - c[2]) ** 2
        r = float(lf.disk_r[v])
        return ok & (dist2 < r * r), 1.0 - torch.sqrt(dist2) / r
    R = lf.poses[v, :9].reshape(3, 3)
    cn = lf.disk_c[v].astype(np.float64) - o
    den = R[0, 2] * d[0] + R[1, 2] * d[1] + R[2, 2] * d[2]
    t = float(R[:, 2] @ cn) / den
    u = t * (R[0, 0] * d[0] + R[1, 0] * d[1] + R[2, 0] * d[2]) - float(R[:, 0] @ cn)
    w = t * (R[0, 1] * d[0] + R[1, 1] * d[1] + R[2, 1] * d[2]) - float(R[:, 1] @ cn)
    e = [float(x) for x in lf.disk_ext[v]]
    rho = torch.sqrt((u / torch.where(u >= 0, e[0], e[1])) ** 2 + (w / torch.where(w >= 0, e[2], e[3])) ** 2)
    return (t >= 0) & (rho < 1.0), 1.0 - rho


def _rays_of(lf, e):
    """World rays of an eye's pixels, their sphere crossings (the far ones) and where these exist."""
    dev, f64 = "cuda", torch.float64
    R, o = e.pose[:9].reshape(3, 3), e.pose[9:]
    ex = ((torch.arange(e.width, device=dev, dtype=f64) + 0.5 - e.intr[2]) / e.intr[0])[None, :].expand(e.height, e.width)
    ey = ((torch.arange(e.height, device=dev, dtype=f64) + 0.5 - e.intr[3]) / e.intr[1])[:, None].expand(e.height, e.width)
    d = [R[k, 0] * ex + R[k, 1] * ey + R[k, 2] for k in range(3)]
    oc = o - lf.sphere_c
    qa = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    qb = d[0] * oc[0] + d[1] * oc[1] + d[2] * oc[2]
    disc = qb * qb - qa * (oc @ oc - lf.sphere_r ** 2)
    t = (torch.sqrt(disc.clamp(min=0.0)) - qb) / qa
    return ex, ey, d, o, [o[k] + t * d[k] for k in range(3)], (disc >= 0) & (t >= 0)


def _exact_eye(st, e, drawn=None):
    """One eye in 64 bits by the method's definition: vertices snapped to 1/256 pixel, the top-left rule,
    the nearest fragment of each view, its bilinear texel under the linear disk weight.  Triangles that
    reach behind the near plane are left out: in these rigs none of them falls into the image."""
    lf, dev, f64 = st.lf, "cuda", torch.float64
    G, W, H = lf.grid_n, lf.width, lf.height
    ex, ey, d, o, p, ok = _rays_of(lf, e)
    Re = torch.tensor(e.pose[:9].reshape(3, 3), device=dev)
    acc = torch.zeros((e.height, e.width, 3), device=dev, dtype=f64)
    wsum = torch.zeros((e.height, e.width), device=dev, dtype=f64)
    k = torch.arange(G - 1, device=dev)
    at = (k[:, None] * G + k[None, :]).reshape(-1)
    tris = torch.stack([torch.stack([at, at + 1, at + G], -1), torch.stack([at + 1, at + G + 1, at + G], -1)], 1).reshape(-1, 3)
    gx = torch.arange(G, device=dev, dtype=f64) * (W / (G - 1))
    gy = torch.arange(G, device=dev, dtype=f64) * (H / (G - 1))
    for v in range(len(lf.poses)) if drawn is None else drawn:
        inside, weight = _disk_rho(lf, v, d, o, p, ok)
        rows, cols = inside.any(1).nonzero(), inside.any(0).nonzero()
        if not len(rows):
            continue
        y0, y1, x0, x1 = int(rows[0]), int(rows[-1]), int(cols[0]), int(cols[-1])
        Rv, tv, K = torch.tensor(lf.poses[v, :9].reshape(3, 3), device=dev), lf.poses[v, 9:], lf.intr[v]
        z = st.depth[v]
        X = torch.stack([z * ((gx - K[2]) / K[0])[None, :], z * ((gy - K[3]) / K[1])[:, None], z], -1).reshape(-1, 3)
        X = (X @ Rv.T + torch.tensor(tv - o, device=dev)) @ Re
        front = X[:, 2] >= Z_NEAR
        zs = torch.where(front, X[:, 2], 1.0)
        sx = torch.round(256.0 * (e.intr[0] * X[:, 0] / zs + e.intr[2])).clamp(-2.0 ** 40, 2.0 ** 40).to(torch.int64)
        sy = torch.round(256.0 * (e.intr[1] * X[:, 1] / zs + e.intr[3])).clamp(-2.0 ** 40, 2.0 ** 40).to(torch.int64)
        TX, TY = sx[tris], sy[tris]
        bx0 = torch.clamp((TX.amin(1) + 127) // 256, min=x0)
        bx1 = torch.clamp((TX.amax(1) - 128) // 256, max=x1)
        by0 = torch.clamp((TY.amin(1) + 127) // 256, min=y0)
        by1 = torch.clamp((TY.amax(1) - 128) // 256, max=y1)
        area = (TX[:, 1] - TX[:, 0]) * (TY[:, 2] - TY[:, 0]) - (TX[:, 2] - TX[:, 0]) * (TY[:, 1] - TY[:, 0])
        keep = (front[tris].all(1) & (area != 0) & (bx0 <= bx1) & (by0 <= by1)
                & (torch.maximum(TX.abs().amax(1), TY.abs().amax(1)) < 2 ** 29)).nonzero()[:, 0]
        if not len(keep):
            continue
        flip = (area[keep] < 0)[:, None]
        TX, TY = torch.where(flip, TX[keep].flip(1), TX[keep]), torch.where(flip, TY[keep].flip(1), TY[keep])
        bx0, by0, bw, bh = bx0[keep], by0[keep], (bx1 - bx0 + 1)[keep], (by1 - by0 + 1)[keep]
        V = X[tris[keep]]
        nrm = torch.linalg.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
        dd = (nrm * V[:, 0]).sum(1)
        n = bw * bh
        which = torch.repeat_interleave(torch.arange(len(keep), device=dev), n)
        j = torch.arange(len(which), device=dev) - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
        px, py = bx0[which] + j % bw[which], by0[which] + j // bw[which]
        cov = inside[py, px]
        which, px, py = which[cov], px[cov], py[cov]
        cov = torch.ones_like(px, dtype=torch.bool)
        for a in range(3):
            b = (a + 1) % 3
            DX, DY = TX[:, b] - TX[:, a], TY[:, b] - TY[:, a]
            tl = ((DY < 0) | ((DY == 0) & (DX > 0))).to(torch.int64)
            C = -DX * TY[:, a] + DY * TX[:, a] + tl
            cov &= DX[which] * (256 * py + 128) - DY[which] * (256 * px + 128) + C[which] > 0
        which, px, py = which[cov], px[cov], py[cov]
        rx, ry = ex[py, px], ey[py, px]
        ne = nrm[which, 0] * rx + nrm[which, 1] * ry + nrm[which, 2]
        z = torch.where(ne != 0, dd[which] / ne, -1.0)
        fine = z > 0
        which, px, py, rx, ry, z = which[fine], px[fine], py[fine], rx[fine], ry[fine], z[fine]
        flat = py * e.width + px
        first = torch.full((e.height * e.width,), float("inf"), device=dev, dtype=f64).scatter_reduce_(0, flat, z, "amin")
        win = z == first[flat]
        which, px, py, rx, ry, z, flat = which[win], px[win], py[win], rx[win], ry[win], z[win], flat[win]
        ids = torch.full((e.height * e.width,), 1 << 60, device=dev).scatter_reduce_(0, flat, keep[which], "amin")
        win = keep[which] == ids[flat]
        px, py, rx, ry, z = px[win], py[win], rx[win], ry[win], z[win]
        P = torch.stack([z * rx, z * ry, z], -1)
        P = (P @ Re.T + torch.tensor(o - tv, device=dev)) @ Rv
        seen = P[:, 2] > 0
        px, py, P = px[seen], py[seen], P[seen]
        if v not in st.cache:
            if len(st.cache) * W * H > 1 << 27:
                st.cache.clear()
            st.cache[v] = st.texels(v)
        col = _bilinear(st.cache[v], K[0] * P[:, 0] / P[:, 2] + K[2] - 0.5, K[1] * P[:, 1] / P[:, 2] + K[3] - 0.5)
        w = weight[py, px]
        acc[py, px] += w[:, None] * col
        wsum[py, px] += w
    valid = (wsum > 0)[..., None]
    rgb = torch.where(valid, acc / torch.where(valid, wsum[..., None], 1.0), 0.0)
    return torch.cat([rgb, valid.to(f64)], -1)


def _bilinear(img, u, v):
    H, W = img.shape[:2]
    u, v = u.clamp(-1.0, W), v.clamp(-1.0, H)
    fu, fv = torch.floor(u), torch.floor(v)
    a, b = (u - fu)[:, None], (v - fv)[:, None]
    i0, j0 = fu.to(torch.int64), fv.to(torch.int64)
    i1, j1 = (i0 + 1).clamp(0, W - 1), (j0 + 1).clamp(0, H - 1)
    i0, j0 = i0.clamp(0, W - 1), j0.clamp(0, H - 1)
    return (1 - a) * (1 - b) * img[j0, i0] + a * (1 - b) * img[j0, i1] + (1 - a) * b * img[j1, i0] + a * b * img[j1, i1]


def _network(p, x):
    """f(x) of n x 3 x H x W images, with the flat parameter vector."""
    w1, b1, w2, b2, w3, b3 = torch.split(p, [864, 32, 9216, 32, 864, 3])
    h = F.relu(F.conv2d(x, w1.view(32, 3, 3, 3), b1, padding=1))
    h = F.relu(F.conv2d(h, w2.view(32, 32, 3, 3), b2, padding=1))
    return F.conv2d(h, w3.view(3, 32, 3, 3), b3, padding=1)


def _exact_refine(params, images):
    p = torch.tensor(params, device="cuda").to(torch.float64)
    out = []
    for im in images:
        x = im[..., :3].to(torch.float64)
        y = x + _network(p, x.permute(2, 0, 1)[None])[0].permute(1, 2, 0)
        ok = im[..., 3:] > 0
        out.append(torch.cat([torch.where(ok, y, 0.0), ok.to(torch.float64)], -1))
    return out


def _exact_train(s):
    p = torch.tensor(s.params, device="cuda").to(torch.float64).requires_grad_(True)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for k in range(s.case["steps"]):
        x, t = (a.to(torch.float64) for a in s.pairs[k % len(s.pairs)])
        ok = ((x[..., 3] > 0) & (t[..., 3] > 0)).to(torch.float64)
        count, loss, g = float(ok.sum()), 0.0, torch.zeros_like(p)
        for a in range(x.shape[0]):
            y = x[a, ..., :3].permute(2, 0, 1)
            err = (y + _network(p, y[None])[0] - t[a, ..., :3].permute(2, 0, 1)) * ok[a]
            part = err.square().sum() / (3.0 * max(count, 1.0))
            g += torch.autograd.grad(part, p)[0]
            loss += float(part.detach())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        step = TRAIN_LR * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)
        p = (p.detach() - step).requires_grad_(True)
    return {"params": p.detach(), "grad": g, "m": m, "v": v, "step": None, "loss": loss}


def _exact_levels(s):
    lf, c = s.lf, s.case
    st = _stored(lf)
    fine, n = c["fine"], c["fine"] + c["coarse"]
    dist = np.linalg.norm(lf.disk_c[fine:, None].astype(float) - lf.disk_c[None, :fine].astype(float), axis=2)
    overlap = dist < lf.disk_r[fine:, None].astype(float) + lf.disk_r[None, :fine].astype(float)
    resident = np.zeros(fine, bool)
    resident[s.first] = True
    images = []
    for e in _level_eyes(s, 0):
        _, _, d, o, p, ok = _rays_of(lf, e)
        seen = np.array([bool(_disk_rho(lf, v, d, o, p, ok)[0].any()) for v in range(n)])
        missing = seen[:fine] & ~resident
        drawn = list(np.flatnonzero(seen[:fine] & resident))
        drawn += [fine + k for k in range(c["coarse"]) if seen[fine + k] and (overlap[k] & missing).any()]
        images.append(_exact_eye(st, e, drawn))
    return {"images": images, "wanted": None, "pages": None}


def _exact_prefilter(s):
    """Eq. 5 with the renders of the dense model read at each mesh point's projection."""
    lf, c, dev, f64 = s.lf, s.case, "cuda", torch.float64
    G, W, H = lf.grid_n, lf.width, lf.height
    st, dense = _stored(lf), _stored(s.dense)
    rho = _sample_weights(s.samples)
    out = []
    for v in range(s.view, s.view + c["block"]):
        R, t, K = lf.poses[v, :9].reshape(3, 3), lf.poses[v, 9:], lf.intr[v]
        nrm = lf.disk_c[v].astype(float) - lf.sphere_c
        nrm /= np.linalg.norm(nrm)
        ax = R[:, 0] - (R[:, 0] @ nrm) * nrm
        ax /= np.linalg.norm(ax)
        ay = np.cross(nrm, ax)
        z = st.depth[v]
        gx = torch.arange(G, device=dev, dtype=f64) * (W / (G - 1))
        gy = torch.arange(G, device=dev, dtype=f64) * (H / (G - 1))
        X = torch.stack([z * ((gx - K[2]) / K[0])[None, :], z * ((gy - K[3]) / K[1])[:, None], z], -1)
        num = torch.zeros((H * W, 4), device=dev, dtype=f64)
        for (a, b, ds, dt), w in zip(s.samples.astype(float), rho):
            th = 2.0 * math.asin(min(1.0, float(lf.disk_r[v]) * math.sqrt(a) / (2.0 * lf.sphere_r)))
            ph = 2.0 * math.pi * b
            o = lf.sphere_c + (1.0 - 1e-5) * lf.sphere_r * (
                math.cos(th) * nrm + math.sin(th) * (math.cos(ph) * ax + math.sin(ph) * ay))
            img = _exact_eye(dense, SimpleNamespace(pose=_pose(R, o), intr=K, width=W, height=H))
            img[..., :3] *= img[..., 3:]
            u = (torch.arange(W, device=dev, dtype=f64) + 0.5 + ds).clamp(0, W)[None, :].expand(H, W).reshape(-1)
            q = (torch.arange(H, device=dev, dtype=f64) + 0.5 + dt).clamp(0, H)[:, None].expand(H, W).reshape(-1)
            cu, cq = u * (G - 1) / W, q * (G - 1) / H
            j, k = cu.floor().clamp(0, G - 2).to(torch.int64), cq.floor().clamp(0, G - 2).to(torch.int64)
            up = (cu - j + cq - k > 1.0).to(torch.int64)
            A, B, C = X[k, j + up], X[k + up, j + 1], X[k + 1, j]
            n = torch.linalg.cross(B - A, C - A)
            rx, ry = (u - K[2]) / K[0], (q - K[3]) / K[1]
            ne = n[:, 0] * rx + n[:, 1] * ry + n[:, 2]
            zz = (n * A).sum(1) / ne
            P = torch.stack([zz * rx, zz * ry, zz], -1) - torch.tensor((o - t) @ R, device=dev)
            ok = (ne != 0) & (P[:, 2] > 0)
            pz = torch.where(ok, P[:, 2], 1.0)
            col = _bilinear(img, K[0] * P[:, 0] / pz + K[2] - 0.5, K[1] * P[:, 1] / pz + K[3] - 0.5)
            num += torch.where(ok[:, None], w * col, 0.0)
        valid = num[:, 3:] > 0
        rgb = torch.where(valid, num[:, :3] / torch.where(valid, num[:, 3:], 1.0), 0.0)
        out.append(torch.cat([rgb, valid.to(f64)], -1).view(H, W, 4))
    return torch.stack(out)


def exact(case, seed):
    c = case
    s = _make(c, seed)
    if c["kind"] == "render":
        st = _stored(s.lf, c["tex"], c["mesh"])
        heads = [[_exact_eye(st, e) for e in head] for head in s.heads]
        if c["form"] in ("host", "refined"):
            heads = [_exact_refine(s.params, head) for head in heads]
        return heads[0][0] if c["form"] == "static" else heads if c["form"] == "host" else heads[0]
    if c["kind"] == "batch":
        st = _stored(s.lf, c["tex"])
        return torch.cat([_exact_eye(st, e).view(-1, 4) for e in s.eyes])
    if c["kind"] == "levels":
        return _exact_levels(s)
    if c["kind"] == "prefilter":
        return _exact_prefilter(s)
    if c["kind"] == "refine":
        return torch.stack(_exact_refine(s.params, s.images))
    return _exact_train(s)

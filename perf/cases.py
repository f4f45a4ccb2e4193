"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is one call (or one replay, or one burst of requests) of a public entry
point on a seeded scene: a room shell with a jointed robot (the renderer's
standard workload), a cube of Gaussians (the small scene), or a room with one
object per environment (the mixed-resolution batch).  ``exact`` renders the
same inputs in 64 bits with plain torch, for the cases where that takes
seconds.
"""
import math

import numpy as np
import torch

from paper_2604_25459_gb300 import gsbatch, synth

DEV = "cuda"
TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
# the resolutions of the mixed batch and the shares of its environments that use them
MIX = ((64, 64, 0.3), (128, 128, 0.3), (320, 240, 0.2), (640, 480, 0.2))


def _case(name, kind, envs, w, h, scene="room", n_bg=500_000, links=20, per_link=5000, dtype="f32", degree=3, rays=0):
    c = dict(kind=kind, envs=envs, w=w, h=h, scene=scene, n_bg=n_bg, links=links, per_link=per_link, dtype=dtype,
             degree=degree, rays=rays)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one view of a small scene (a first script, a unit test, an interactive viewer)
        _case("one_small", "render", 1, 128, 96, scene="cube", n_bg=16_384, links=0, per_link=0),
        # a control loop that may not allocate: a few views of a small scene in the library's fixed array
        _case("control_noalloc", "noalloc", 8, 128, 96, scene="cube", n_bg=16_384, links=0, per_link=0),
        # evaluating one policy: a single robot in the full room, RGB, depth and alpha at camera resolution
        _case("one_room_vga", "render", 1, 640, 480),
        # a small evaluation batch at an odd resolution, attributes stored in 16 bits
        _case("eval_ragged_f16", "render", 16, 333, 251, dtype="f16"),
        # training step of a vectorised environment: 8-bit RGB after appearance randomisation and half depth
        _case("train_obs_128", "obs", 512, 128, 128),
        # the headline batch at a quarter of a training job's environments: full room at 640x480
        _case("train_room_vga", "render", 256, 640, 480),
        # the same kind of step for a simulator that lives on the host: pinned host poses in, images out
        _case("host_step_128", "host", 128, 128, 128),
        # many tasks at once: mixed resolutions, one object per environment, a tuned plan replayed as a graph
        _case("plan_mixed", "plan", 256, 640, 480, scene="objects", n_bg=300_000, links=256, per_link=60_000),
        # rendering as a service: a burst of single-environment requests over two resident scenes
        _case("serve_burst", "serve", 128, 640, 480, n_bg=200_000),
        # a spinning LiDAR per environment
        _case("lidar_spin", "lidar", 32, 1024, 64),
        # a non-repetitive LiDAR pattern per environment, given as a list of rays
        _case("lidar_rosette", "rays", 32, 256, 256, rays=20_011),
        # ranking the Gaussians before a scene is pruned: summed blending weights over sampled views
        _case("prune_scores", "contribution", 16, 640, 480),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["render", "render", "obs", "lidar", "rays", "contribution", "host", "plan", "noalloc", "serve"])
    dtype = rng.choice(["f32", "f32", "bf16", "f16"])
    degree = rng.choice([3, 3, 3, 2, 1, 0])
    if kind == "noalloc":  # sizes that the fixed array holds
        w = _log(rng, 16, 128)
        return _case(None, kind, _log(rng, 1, 24), w, max(8, min(96, w * 3 // 4 + rng.randint(-5, 5))), scene="cube",
                     n_bg=_log(rng, 500, 16_384), links=0, per_link=0, dtype=dtype, degree=degree)
    if kind == "serve":
        return _case(None, kind, _log(rng, 8, 128), 640, 480, n_bg=_log(rng, 50_000, 200_000))
    if kind == "plan":
        e = _log(rng, 8, 192)
        return _case(None, kind, e, 640, 480, scene="objects", n_bg=_log(rng, 20_000, 300_000), links=e,
                     per_link=_log(rng, 5_000, 60_000), dtype=dtype)
    n_bg, per = _log(rng, 5_000, 500_000), _log(rng, 200, 5_000)
    if kind == "lidar":
        return _case(None, kind, _log(rng, 1, 32), _log(rng, 90, 1024), _log(rng, 8, 64), n_bg=n_bg, per_link=per)
    if kind == "rays":
        return _case(None, kind, _log(rng, 1, 32), 256, 256, n_bg=n_bg, per_link=per, rays=_log(rng, 500, 20_000))
    w = _log(rng, 40, 640)
    h = max(30, min(480, int(w * rng.uniform(0.6, 1.0))))
    most = {"render": 256, "obs": 512, "host": 128, "contribution": 16}[kind]
    return _case(None, kind, _log(rng, 1, most if w <= 128 else max(2, most // 4)), w, h, n_bg=n_bg, per_link=per,
                 dtype=dtype, degree=degree)


# ------------------------------------------------------------------ inputs


class _G:
    """A set of Gaussians as the scene takes it (CUDA tensors)."""

    def __init__(self, mean, quat, log_scale, opacity, sh):
        self.mean, self.quat, self.log_scale, self.opacity, self.sh = mean, quat, log_scale, opacity, sh


def _attributes(gen, mean, dtype, degree):
    n, nk, t = mean.shape[0], (degree + 1) ** 2, TYPES[dtype]
    r = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    q = r(n, 4)
    sh = 0.3 * r(n, nk, 3)
    sh[:, 0] += 0.5
    return _G(mean.float().contiguous(), q / q.norm(dim=1, keepdim=True), (r(n, 3) * 0.5 - 4.0).to(t),
              torch.sigmoid(r(n)).to(t), sh.to(t).contiguous())


def _room(gen, n):
    """n means area-uniform on the faces of a 10 x 10 x 3 m room, jittered along the face normal."""
    ext = torch.tensor([10.0, 10.0, 3.0], device=DEV)
    face = torch.multinomial(torch.tensor([30.0, 30, 30, 30, 100, 100], device=DEV), n, True, generator=gen)
    axis, side = face // 2, (face % 2).float()
    p = torch.rand(n, 3, generator=gen, device=DEV)
    p.scatter_(1, axis[:, None], side[:, None])
    m = (p - torch.tensor([0.5, 0.5, 0.0], device=DEV)) * ext
    off = 0.02 * torch.randn(n, 1, generator=gen, device=DEV)
    return m.scatter_add_(1, axis[:, None], off)


def _inputs(case, seed):
    """Gaussians, cameras and poses of a case: everything but the framework's own objects."""
    gen = torch.Generator(device=DEV).manual_seed(seed * 7919 + 17)
    rng = np.random.default_rng([seed, 3])
    c, E, L = case, case["envs"], case["links"]
    att = lambda m: _attributes(gen, m, c["dtype"], c["degree"])
    r = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    inp = {}
    if c["scene"] == "cube":
        inp["bg"] = att(torch.rand(c["n_bg"], 3, generator=gen, device=DEV) * 2 - 1)
        t = np.concatenate([rng.uniform(-0.2, 0.2, (E, 2)), np.full((E, 1), 3.0)], 1)
        f = 110.0 * c["w"] / 128
        inp["cams"] = synth.make_cameras(E, f, f, c["w"] / 2, c["h"] / 2, c["w"], c["h"], [[1, 0, 0, 0]] * E, t)
        inp["offsets"], inp["links"], inp["poses"] = np.zeros(1, np.int64), None, np.zeros((E, 0, 7), np.float32)
        return inp
    inp["bg"] = att(_room(gen, c["n_bg"]))
    if c["scene"] == "objects":  # one object per environment, sizes log-uniform about per_link
        sizes = np.exp(rng.uniform(np.log(c["per_link"] / 5), np.log(c["per_link"] * 2), L)).astype(np.int64)
        inp["offsets"] = np.concatenate([[0], np.cumsum(sizes)])
        inp["links"] = att(0.15 * r(int(inp["offsets"][-1]), 3))
        q = rng.normal(size=(L, 4))
        pos = np.stack([0.6 + rng.uniform(-0.2, 0.2, L), rng.uniform(-0.3, 0.3, L), 0.6 + rng.uniform(0, 0.3, L)], 1)
        inp["poses"] = np.concatenate([q / np.linalg.norm(q, axis=1, keepdims=True), pos], 1).astype(np.float32)
    else:
        inp["offsets"] = np.arange(L + 1, dtype=np.int64) * c["per_link"]
        inp["links"] = att(0.05 * r(L * c["per_link"], 3))
        inp["poses"] = synth.chain_link_poses(rng.uniform(-1, 1, (E, L)))
    s = int(rng.integers(1 << 30))
    if c["kind"] in ("plan", "serve"):
        res = np.random.default_rng(E).choice(len(MIX), size=E, p=[m[2] for m in MIX])  # the same for every seed
        cams = np.zeros(E, synth.CAMERA_DTYPE)
        for k, (w, h, _) in enumerate(MIX):
            cams[res == k] = synth.head_cameras(E, s, w, h, synth.focal_for(w, h))[res == k]
        inp["cams"] = cams
    elif c["kind"] in ("lidar", "rays"):
        wide = c["kind"] == "lidar"
        d = np.zeros(E, gsbatch.LIDAR_DTYPE)
        yaw = rng.uniform(-0.2, 0.2, E)
        pos = np.array([-1.0, 0.0, 1.4]) + rng.uniform(-0.2, 0.2, (E, 3))
        d["q_ws"] = np.stack([np.cos(yaw / 2), 0 * yaw, 0 * yaw, -np.sin(yaw / 2)], 1)
        cy, sy = np.cos(yaw), np.sin(yaw)
        d["t_ws"] = -np.stack([cy * pos[:, 0] + sy * pos[:, 1], -sy * pos[:, 0] + cy * pos[:, 1], pos[:, 2]], 1)
        d["rows"], d["cols"], d["near_range"] = c["h"], c["w"], 0.05
        d["elev_min"], d["elev_max"] = (-0.4, 0.3) if wide else (-0.65, 0.65)
        d["az_min"], d["az_max"] = (0.0, 2 * math.pi) if wide else (-0.65, 0.65)
        inp["sensors"] = d
        if not wide:
            inp["dirs"] = synth.rosette_rays(E, c["rays"], s)
    else:
        inp["cams"] = synth.head_cameras(E, s, c["w"], c["h"], 500.0 * c["w"] / 640)
    if c["kind"] == "obs":
        inp["appear"] = np.stack([rng.uniform(-0.5, 0.5, E), rng.uniform(0.8, 1.2, E), rng.uniform(-0.1, 0.1, E)],
                                 1).astype(np.float32)
    if c["kind"] == "serve":  # the second resident scene has a background five times as large
        inp["bg2"] = att(_room(gen, 5 * c["n_bg"]))
    return inp


def _scene(case, inp, bg="bg"):
    def stored(g):
        return None if case["dtype"] == "f32" else dict(log_scale=g.log_scale, opacity=g.opacity, sh=g.sh)

    s = gsbatch.Scene(inp[bg], case["dtype"], case["degree"], stored=stored(inp[bg]))
    if inp["links"] is not None:
        s.attach_links(inp["offsets"], inp["links"], stored=stored(inp["links"]))
    return s


def prepare(case, seed):
    inp, E, W, H, kind = _inputs(case, seed), case["envs"], case["w"], case["h"], case["kind"]
    st = {"case": case, "scene": _scene(case, inp), "cams": inp.get("cams")}
    st["poses"] = torch.from_numpy(inp["poses"]).to(DEV) if inp["poses"].size else None
    new = lambda *s, t=torch.float32: torch.zeros(*s, dtype=t, device=DEV)
    if kind in ("render", "noalloc"):
        st["out"] = (new(E, H, W, 3), new(E, H, W), new(E, H, W))
    elif kind == "obs":
        st["appear"] = torch.from_numpy(inp["appear"]).to(DEV)
        st["out"] = (new(E, H, W, 3, t=torch.uint8), new(E, H, W, t=torch.float16))
    elif kind == "host":
        pin = lambda *s: torch.zeros(*s).pin_memory().numpy()
        st["poses"] = torch.from_numpy(inp["poses"]).pin_memory().numpy()
        st["out"] = (pin(E, H, W, 3), pin(E, H, W))
    elif kind in ("lidar", "rays"):
        st["sensors"] = inp["sensors"]
        shape = (E, H, W) if kind == "lidar" else (E, case["rays"])
        st["out"] = (new(*shape), new(*shape))
        if kind == "rays":
            st["dirs"] = torch.from_numpy(inp["dirs"]).to(DEV)
    elif kind == "contribution":
        st["out"] = new(case["n_bg"] + case["links"] * case["per_link"])
    elif kind == "plan":
        ids = np.arange(E)
        envs = gsbatch.make_envs(inp["cams"], np.stack([ids, ids + 1], 1), ids)
        px = int((envs["cam"]["width"].astype(np.int64) * envs["cam"]["height"]).sum())
        st["out"] = (new(px, 3), new(px))
        st["plan"] = st["scene"].plan(envs)
        st["plan"].launch(st["poses"], *st["out"])  # the first launch tunes and captures
    elif kind == "serve":
        st["scene2"] = _scene(case, inp, "bg2")
        st["server"] = sv = gsbatch.Server(16 << 30, max_inflight=4, max_batch_envs=64)
        ids = [sv.add_scene(st["scene"]), sv.add_scene(st["scene2"])]
        st["ids"] = [sv.add_env(ids[e % 2], inp["cams"][e:e + 1], 0, case["links"]) for e in range(E)]
        sv.start()
        st["req"] = inp["poses"]
        st["views"] = [sv.env_output(e) for e in st["ids"]]
    return st


def run(st):
    k, sc, poses, out = st["case"]["kind"], st["scene"], st["poses"], st.get("out")
    if k == "render":
        sc.render(poses, st["cams"], *out)
    elif k == "noalloc":
        sc.render_noalloc(poses, st["cams"], *out, stream=torch.cuda.current_stream())
    elif k == "obs":
        sc.render_obs(poses, st["cams"], st["appear"], *out)
    elif k == "host":
        sc.render_host(poses, st["cams"], *out)
    elif k == "lidar":
        sc.render_lidar(poses, st["sensors"], *out)
    elif k == "rays":
        sc.render_rays(poses, st["sensors"], st["dirs"], *out)
    elif k == "contribution":
        sc.contribution(poses, st["cams"], out.zero_())
    elif k == "plan":
        st["plan"].launch(poses, *out)
    else:  # serve: a burst of requests, waited for, their images taken out of the server's memory
        sv = st["server"]
        for e, p in zip(st["ids"], st["req"]):
            sv.submit(e, p)
        sv.drain()
        sv.poll(len(st["ids"]))
        return torch.cat([v[0].view(-1, 3) for v in st["views"]]), torch.cat([v[1].view(-1) for v in st["views"]])
    return out


def _pixels(case):
    """Pixels or rays over all environments (the mixed batch: by its shares)."""
    if case["kind"] in ("plan", "serve"):
        return case["envs"] * sum(w * h * p for w, h, p in MIX)
    return case["envs"] * (case["rays"] or case["w"] * case["h"])


def work(case):
    """Attributes read once, outputs written once; per (environment, Gaussian) pair the cull, and per pixel the
    blending of 20 splats at 20 operations (rooms blend 58 per pixel, small views fewer)."""
    width = 4 if case["dtype"] == "f32" else 2
    n = case["n_bg"] * (6 if case["kind"] == "serve" else 1) + case["links"] * case["per_link"]
    seen = case["n_bg"] + (case["per_link"] if case["scene"] == "objects" else case["links"] * case["per_link"])
    px = _pixels(case)
    per = {"render": 20, "noalloc": 20, "obs": 5, "host": 16, "plan": 16, "serve": 16, "lidar": 8, "rays": 20}
    out = 4 * n if case["kind"] == "contribution" else per[case["kind"]] * px
    return {"bytes": n * (28 + width * (4 + 3 * (case["degree"] + 1) ** 2)) + 28 * case["envs"] * case["links"] + out,
            "flops": case["envs"] * seen * 40 + px * 800}


# ------------------------------------------------------------------ the same in 64 bits, plain torch

_PIX = 24  # pixels along the side of a block rendered at once
_K = 4096  # splats composited at once


def _rot(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).view(*q.shape[:-1], 3, 3)


class _World:
    """A case's Gaussians in 64 bits, with their link (0: background)."""

    def __init__(self, inp, bg="bg"):
        gs = [inp[bg]] + ([inp["links"]] if inp["links"] is not None else [])
        cat = lambda f: torch.cat([getattr(g, f).double() for g in gs])
        self.mean, self.o, self.sh = cat("mean"), cat("opacity"), cat("sh")
        self.scale, self.R = cat("log_scale").exp(), _rot(cat("quat"))
        off = torch.from_numpy(inp["offsets"]).to(DEV)
        link = torch.zeros(len(self.o), dtype=torch.long, device=DEV)
        if len(off) > 1:
            link[len(inp[bg].mean):] = torch.repeat_interleave(torch.arange(1, len(off), device=DEV), off.diff())
        self.link = link

    def select(self, link):
        s = object.__new__(_World)
        m = (self.link == 0) | (self.link == link)
        for f in ("mean", "o", "sh", "scale", "R", "link"):
            setattr(s, f, getattr(self, f)[m])
        s.link = (s.link > 0).long()
        return s

    def frames(self, q, t, poses):
        """Per link (0: world) the transform into the view and the view's centre there."""
        d = lambda a: torch.from_numpy(np.asarray(a, np.float32).astype(np.float64)).to(DEV)
        Rc, tc = _rot(d(q)), d(t)
        R, T = [Rc], [tc]
        if len(poses):
            p = d(poses)
            Rl = _rot(p[:, :4])
            R += list(Rc @ Rl)
            T += list(p[:, 4:] @ Rc.T + tc)
        R, T = torch.stack(R), torch.stack(T)
        return R, T, -(R.transpose(1, 2) @ T[..., None])[..., 0]


def _sh_colour(sh, d):
    x, y, z = d.unbind(-1)
    xx, yy, zz = x * x, y * y, z * z
    p = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(p))]
    if sh.shape[1] > 1:
        a = math.sqrt(3 / (4 * p))
        Y += [-a * y, a * z, -a * x]
    if sh.shape[1] > 4:
        a, b = math.sqrt(15 / (4 * p)), math.sqrt(5 / (16 * p))
        Y += [a * x * y, -a * y * z, b * (2 * zz - xx - yy), -a * x * z, a / 2 * (xx - yy)]
    if sh.shape[1] > 9:
        a, b, c, e = math.sqrt(35 / (32 * p)), math.sqrt(105 / (4 * p)), math.sqrt(21 / (32 * p)), math.sqrt(7 / (16 * p))
        Y += [-a * y * (3 * xx - yy), b * x * y * z, -c * y * (4 * zz - xx - yy), e * z * (2 * zz - 3 * xx - 3 * yy),
              -c * x * (4 * zz - xx - yy), b / 2 * z * (xx - yy), -a * x * (xx - 3 * yy)]
    return ((torch.stack(Y, 1)[:, :, None] * sh).sum(1) + 0.5).clamp_min(0)


def _blend(alpha_of, idx, n_px, value, weights=None):
    """Front-to-back compositing of the ordered splats idx over n_px pixels; alpha_of(idx) -> [px, k] alphas and
    per-pair values (or None: value[idx]).  Returns sum(alpha T value) and T."""
    T = torch.ones(n_px, dtype=torch.double, device=DEV)
    acc = torch.zeros(n_px, value.shape[1] if value is not None else 1, dtype=torch.double, device=DEV)
    live = torch.ones(n_px, dtype=torch.bool, device=DEV)
    for k in range(0, len(idx), _K):
        i = idx[k:k + _K]
        al, val = alpha_of(i)
        al = torch.where(al >= 1 / 255, al.clamp_max(0.99), 0.0)
        c = T[:, None] * torch.cumprod(1 - al, 1)
        ok = (c >= 1e-4) & live[:, None]
        w = torch.where(ok, al * torch.cat([T[:, None], c[:, :-1]], 1), 0.0)
        acc += w @ value[i] if val is None else (w * val).sum(1, keepdim=True)
        if weights is not None:
            weights.index_add_(0, i, w.sum(0))
        T = torch.where(ok, c, T[:, None]).amin(1)
        live = ok[:, -1]
        if not bool(live.any()):
            break
    return acc, T


def _exact_camera(world, cam, poses, weights=None):
    W, H = int(cam["width"]), int(cam["height"])
    fx, fy, cx, cy = (float(cam[k]) for k in ("fx", "fy", "cx", "cy"))
    R, T, O = world.frames(cam["q_cw"], cam["t_cw"], poses)
    ln = world.link
    p = (R[ln] @ world.mean[..., None])[..., 0] + T[ln]
    keep = ((p[:, 2] > float(cam["near_plane"])) & (world.o >= 1 / 255)).nonzero()[:, 0]
    p, ln = p[keep], ln[keep]
    z = p[:, 2]
    u, v = fx * p[:, 0] / z + cx, fy * p[:, 1] / z + cy
    tx = (p[:, 0] / z).clamp(-1.3 * cx / fx, 1.3 * (W - cx) / fx)
    ty = (p[:, 1] / z).clamp(-1.3 * cy / fy, 1.3 * (H - cy) / fy)
    J = torch.zeros(len(z), 2, 3, dtype=torch.double, device=DEV)
    J[:, 0, 0], J[:, 0, 2], J[:, 1, 1], J[:, 1, 2] = fx / z, -fx * tx / z, fy / z, -fy * ty / z
    M = J @ R[ln] @ (world.R[keep] * world.scale[keep][:, None, :])
    A, C, B = (M[:, 0] ** 2).sum(1) + 0.3, (M[:, 1] ** 2).sum(1) + 0.3, (M[:, 0] * M[:, 1]).sum(1)
    det = (torch.linalg.cross(M[:, 0], M[:, 1]) ** 2).sum(1) + 0.3 * (A + C - 0.6) + 0.09
    o = world.o[keep]
    qs = 2 * torch.log(255 * o)
    hx, hy = (qs * A).sqrt() * 1.0001, (qs * C).sqrt() * 1.0001
    d = world.mean[keep] - O[ln]
    val = torch.cat([_sh_colour(world.sh[keep], d / d.norm(dim=1, keepdim=True)), z[:, None]], 1)
    order = torch.argsort(z, stable=True)
    inside = (u + hx > 0) & (u - hx < W) & (v + hy > 0) & (v - hy < H)
    order = order[inside[order]]
    rgb = torch.zeros(H, W, 3, dtype=torch.double, device=DEV)
    dep, alp = torch.zeros(H, W, dtype=torch.double, device=DEV), torch.zeros(H, W, dtype=torch.double, device=DEV)
    uo, vo, hxo, hyo = u[order], v[order], hx[order], hy[order]
    wk = None if weights is None else torch.zeros(len(z), dtype=torch.double, device=DEV)
    for y0 in range(0, H, _PIX):
        y1 = min(H, y0 + _PIX)
        row = order[(vo + hyo > y0) & (vo - hyo < y1)]
        ur, hr = u[row], hx[row]
        for x0 in range(0, W, _PIX):
            x1 = min(W, x0 + _PIX)
            idx = row[(ur + hr > x0) & (ur - hr < x1)]
            yy, xx = torch.meshgrid(torch.arange(y0, y1, device=DEV) + 0.5, torch.arange(x0, x1, device=DEV) + 0.5,
                                    indexing="ij")
            px, py = xx.reshape(-1, 1).double(), yy.reshape(-1, 1).double()

            def alphas(i):
                dx, dy = px - u[i], py - v[i]
                q = (C[i] * dx * dx - 2 * B[i] * dx * dy + A[i] * dy * dy) / det[i]
                return o[i] * torch.exp(-0.5 * q), None

            acc, Tn = _blend(alphas, idx, len(px), val, wk)
            a = 1 - Tn
            rgb[y0:y1, x0:x1] = acc[:, :3].clamp(0, 1).view(y1 - y0, x1 - x0, 3)
            dep[y0:y1, x0:x1] = torch.where(a > 0, acc[:, 3] / a.clamp_min(1e-300), 0.0).view(y1 - y0, x1 - x0)
            alp[y0:y1, x0:x1] = a.view(y1 - y0, x1 - x0)
    if weights is not None:
        weights.index_add_(0, keep, wk)
    return rgb, dep, alp


def _exact_rays(world, sensor, poses, dirs):
    """Scan along unit directions [n, 3] (64 bits), 256 neighbouring ones at a time."""
    R, T, _ = world.frames(sensor["q_ws"], sensor["t_ws"], poses)
    ln = world.link
    mu = (R[ln] @ world.mean[..., None])[..., 0] + T[ln]
    dist = mu.norm(dim=1)
    keep = world.o >= 1 / 255
    order = torch.argsort(dist, stable=True)
    order = order[keep[order]]
    G = ((R[ln] @ world.R) / world.scale[:, None, :]).transpose(1, 2)  # rows e^-s_k r_k
    b = (G @ mu[..., None])[..., 0]
    reach = (2 * torch.log(255 * world.o.clamp_min(1 / 255))).sqrt() * world.scale.amax(1)
    spread = torch.asin((reach / dist.clamp_min(1e-12)).clamp_max(1.0)) + 1e-6
    spread[reach >= dist] = 4.0
    unit, o, near = mu / dist.clamp_min(1e-12)[:, None], world.o, float(sensor["near_range"])
    rng, hit = (torch.zeros(len(dirs), dtype=torch.double, device=DEV) for _ in range(2))
    uo, so = unit[order], spread[order]
    for k in range(0, len(dirs), 256):
        d = dirs[k:k + 256]
        c = d.mean(0)
        c = c / c.norm()
        half = torch.acos((d @ c).clamp(-1, 1)).max()
        idx = order[torch.acos((uo @ c).clamp(-1, 1)) <= so + half + 1e-6]

        def alphas(i):
            a = torch.einsum("kij,pj->pki", G[i], d)
            aa, ab = (a * a).sum(-1), (a * b[i]).sum(-1)
            cr = torch.linalg.cross(a, b[i].expand_as(a))
            t = ab / aa
            return torch.where(t > near, o[i] * torch.exp(-0.5 * (cr * cr).sum(-1) / aa), 0.0), t

        acc, Tn = _blend(alphas, idx, len(d), None)
        hit[k:k + 256] = 1 - Tn
        rng[k:k + 256] = torch.where(Tn < 1, acc[:, 0] / (1 - Tn).clamp_min(1e-300), 0.0)
    return rng, hit


def exact(case, seed):
    kind, E = case["kind"], case["envs"]
    views = E * (case["n_bg"] + case["links"] * case["per_link"] if case["scene"] != "objects" else case["n_bg"])
    if kind == "serve" or _pixels(case) > 8e6 or views > (2e7 if kind in ("lidar", "rays") else 8e7):
        return None  # more than some seconds of 64-bit arithmetic
    inp = _inputs(case, seed)
    world, poses = _World(inp), inp["poses"]
    if kind == "contribution":
        w = torch.zeros(len(world.o), dtype=torch.double, device=DEV)
        for e in range(E):
            _exact_camera(world, inp["cams"][e], poses[e], w)
        return w
    if kind in ("lidar", "rays"):
        out = []
        for e in range(E):
            s, W, H = inp["sensors"][e], case["w"], case["h"]
            if kind == "rays":
                d = torch.from_numpy(inp["dirs"][e].astype(np.float64)).to(DEV)
                d = d / d.norm(dim=1, keepdim=True)
                cell = (torch.asin(d[:, 2]) / 0.05).floor() * 1000 + torch.atan2(d[:, 1], d[:, 0]) / 0.05
                perm = torch.argsort(cell)
            else:
                phi = float(s["az_min"]) + (float(s["az_max"]) - float(s["az_min"])) * (torch.arange(W, device=DEV).double() + 0.5) / W
                th = float(s["elev_min"]) + (float(s["elev_max"]) - float(s["elev_min"])) * (torch.arange(H, device=DEV).double() + 0.5) / H
                th, phi = (t.reshape(-1) for t in torch.meshgrid(th, phi, indexing="ij"))
                d = torch.stack([th.cos() * phi.cos(), th.cos() * phi.sin(), th.sin()], 1)
                j = torch.arange(H * W, device=DEV)
                perm = torch.argsort((j // W // 16) * (W * 16) + (j % W) // 16 * 16, stable=True)
            r, h = _exact_rays(world, s, poses[e], d[perm])
            back = torch.argsort(perm)
            out.append((r[back], h[back]))
        shape = (H, W) if kind == "lidar" else (-1,)
        return tuple(torch.stack([o[k].view(shape) for o in out]) for k in range(2))
    if kind == "plan":
        imgs = [_exact_camera(world.select(e + 1), inp["cams"][e], poses[e:e + 1]) for e in range(E)]
        return torch.cat([i[0].view(-1, 3) for i in imgs]), torch.cat([i[1].view(-1) for i in imgs])
    imgs = [_exact_camera(world, inp["cams"][e], poses[e]) for e in range(E)]
    out = tuple(torch.stack([i[k] for i in imgs]) for k in range(3))
    if kind == "obs":
        return None, out[1]
    return tuple(x.cpu().numpy() for x in out[:2]) if kind == "host" else out

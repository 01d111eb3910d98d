"""The work that a user of this library has it do, as cases to time and to compare.

A case is a dict of plain values; `prepare` makes what a mapping program holds before the call
(map, keyframes, targets, moments, workspace, captured graph), `run` is one pass through the
public entry points, `work` the bytes and operations that the path cannot do without, `exact`
the same results in 64 bits from plain torch.

The scenes are made on the GPU from the seed alone: a 32-beam spinning LiDAR driven along a
40 m line or a 200 m loop past box facades on a ground plane (one Gaussian per return, in scan
order), with cameras at trajectory poses whose target images are ray casts of the same
surfaces.  Pixels that see no surface within range have no depth reference, as with a LiDAR.

Every optimising step starts from the map kept in the state (one copy of the parameters inside
`run`): repeated passes then work on the same map however often they are run, as a program does
that rolls back to its last accepted map.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2604_12942_gb300 as gs
from paper_2604_12942_gb300 import learned

DEV = "cuda"
Y00 = 0.28209479177387814
FAR = 60.0                      # m, range of the LiDAR and of the depth references
# Work per pixel of the compositing: about 115 (pixel, Gaussian) evaluations survive the culling
# on LiDAR maps, at 20 operations forward and 60 backward each; about a third of the map's rows
# are seen by a batch.
EVALS, OPS_FWD, OPS_BWD, SEEN = 115, 20, 60, 1 / 3


def listed():
    return [
        # one keyframe of a small fresh map, gradients and pose twist without an update: the
        # smallest call, where launches and latency count
        dict(name="keyframe_10k_grads", kind="step", scene="box", n=10_000, sh=0, sizes="320x240", tile=16, chunk=64,
             mode="grads", objective="l1"),
        # the loop that trains and evaluates the learned initialiser: eager steps over 8 keyframes
        # of 320 x 240 drawn anew (new poses) each iteration, degree-1 colour
        dict(name="loop_200k_8x320", kind="step", scene="line", n=200_000, sh=1, sizes="320x240*8", tile=16, chunk=64,
             mode="eager", objective="l1"),
        # one outdoor keyframe at 1280 x 720, a captured step fed from pinned host buffers
        dict(name="outdoor_500k_720p_host", kind="step", scene="line", n=500_000, sh=3, sizes="1280x720", tile=16,
             chunk=256, mode="host", objective="l1"),
        # the global optimisation: 8 keyframes of uneven size over the 2M-Gaussian map, captured
        dict(name="batch_2M_8views", kind="step", scene="loop", n=2_000_000, sh=3,
             sizes="640x480*2,960x540*2,1280x720*2,1280x1024*2", tile=16, chunk=256, mode="graph", objective="l1"),
        # the paper's full objective (SSIM inside the eroded interior mask), captured
        dict(name="ssim_1M_4views", kind="step", scene="loop", n=1_000_000, sh=3,
             sizes="640x480,960x540,1280x720,1280x1024", tile=16, chunk=256, mode="graph", objective="ssim"),
        # one rank's share of the view-parallel step: gradients, twists, then the separate masked
        # Adam with half of the map frozen
        dict(name="parallel_1M_1024x768", kind="step", scene="loop", n=1_000_000, sh=3, sizes="1024x768*2", tile=16,
             chunk=256, mode="parallel", objective="l1"),
        # any objective through torch.autograd, with pose increments, odd image sizes, degree 2
        dict(name="autograd_100k_odd", kind="autograd", scene="line", n=100_000, sh=2, sizes="853x479,641x363", tile=16,
             chunk=64),
        # rendering without gradients: held-out views, previews
        dict(name="render_2M_8views", kind="render", scene="loop", n=2_000_000, sh=3,
             sizes="640x480*2,960x540*2,1280x720*2,1280x1024*2", tile=16, chunk=64),
        # a new segment's points: voxel features against 16 keyframes, the MLP, the cascade
        dict(name="init_400k", kind="init", n=400_000, frames=16, sh=3),
        # training of the initialiser, one batch
        dict(name="mlp_train_16k", kind="mlp_train", n=16_384),
        # map maintenance between iterations: prune, proximity test, compaction
        dict(name="map_update_2M", kind="map_update", n=2_000_000, new=200_000, sh=3),
        # a loop candidate: target set from 4 query views, registration of a revisited scan
        dict(name="gicp_2M_map", kind="gicp", n=2_000_000, src=80_000),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_sizes(rng, n, views):
    sizes, px = [], 0
    for _ in range(views):
        w = _spread(rng, 160, 1280)
        h = max(120, min(1024, int(w * rng.uniform(0.5, 0.85))))
        if px + w * h > 6_000_000:
            break
        px += w * h
        sizes.append(f"{w}x{h}")
    return ",".join(sizes)


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["autograd", "render", "init", "mlp_train", "map_update", "gicp"])
    if kind in ("step", "autograd", "render"):
        n = _spread(rng, 10_000, 2_000_000 if kind != "autograd" else 300_000)
        views = rng.randint(1, 8 if kind != "autograd" else 3)
        c = dict(kind=kind, scene=rng.choice(["line", "loop", "loop"]), n=n, sh=rng.choice([0, 1, 2, 3, 3, 3]),
                 sizes=_draw_sizes(rng, n, views), tile=rng.choice([16, 16, 16, 8]), chunk=rng.choice([64, 128, 256]))
        if kind == "step":
            c["mode"] = rng.choice(["graph", "graph", "eager", "grads", "parallel", "host"])
            c["objective"] = rng.choice(["l1", "l1", "masked", "ssim"]) if c["mode"] != "parallel" else "l1"
        return c
    if kind == "init":
        return dict(kind=kind, n=_spread(rng, 20_000, 400_000), frames=rng.randint(1, 32), sh=rng.choice([0, 1, 3]))
    if kind == "mlp_train":
        return dict(kind=kind, n=_spread(rng, 1_000, 65_536))
    if kind == "map_update":
        return dict(kind=kind, n=_spread(rng, 50_000, 2_000_000), new=_spread(rng, 1_000, 200_000), sh=rng.choice([0, 1, 3]))
    return dict(kind=kind, n=_spread(rng, 100_000, 2_000_000), src=_spread(rng, 2_000, 80_000))


# -- scenes ------------------------------------------------------------------------------------

def _sizes(case):
    out = []
    for part in case["sizes"].split(","):
        wh, _, k = part.partition("*")
        w, h = wh.split("x")
        out += [(int(w), int(h))] * int(k or 1)
    return out


def _path(scene, s):
    """Sensor position (z = 1.8 m) and heading at s in [0, 1) of the trajectory."""
    if scene == "loop":
        r = 200.0 / (2 * math.pi)
        a = 2 * math.pi * s
        return np.stack([r * np.cos(a), r * np.sin(a), np.full_like(a, 1.8)], -1), a + math.pi / 2
    return np.stack([40.0 * s, np.zeros_like(s), np.full_like(s, 1.8)], -1), np.zeros_like(s)


class _World:
    """Ground plane, box facades and their procedural texture."""

    def __init__(self, scene, seed):
        rs = np.random.RandomState(seed % (1 << 31))
        path, _ = _path(scene, np.linspace(0, 1, 400, endpoint=False))
        self.scene, self.boxes = scene, []
        while len(self.boxes) < 20:
            size = np.array([rs.uniform(2, 20), rs.uniform(2, 20), rs.uniform(3, 20)])
            ang, dist = rs.uniform(0, 2 * math.pi), rs.uniform(6, 36)
            c = path[rs.randint(len(path)), :2] + dist * np.array([math.cos(ang), math.sin(ang)])
            lo, hi = c - size[:2] / 2, c + size[:2] / 2
            clear = np.maximum(np.maximum(lo - path[:, :2], path[:, :2] - hi), 0).max(1).min()
            if clear > 3.0:                                     # a free corridor around the path
                self.boxes.append((*lo, 0.0, *hi, size[2]))
        self.freq = torch.as_tensor(rs.uniform(0.4, 3.0, (3, 3)), dtype=torch.float32, device=DEV)
        self.phase = torch.as_tensor(rs.uniform(0, 2 * math.pi, (3, 3)), dtype=torch.float32, device=DEV)
        self.base = torch.as_tensor(rs.uniform(0.2, 0.8, 3), dtype=torch.float32, device=DEV)

    def cast(self, o, d):
        """Ranges (inf: nothing hit) and the face axis of the rays o + s d; o, d [3, m]."""
        best = torch.where(d[2] < 0, -o[2] / d[2], torch.inf)
        axis = torch.full_like(best, 2, dtype=torch.uint8)
        inv = 1.0 / torch.where(d == 0, 1e-12, d)
        for b in self.boxes:
            lo = torch.tensor(b[:3], dtype=torch.float32, device=DEV)[:, None]
            hi = torch.tensor(b[3:], dtype=torch.float32, device=DEV)[:, None]
            t1, t2 = (lo - o) * inv, (hi - o) * inv
            enter, ax = torch.minimum(t1, t2).max(0)
            hit = (enter <= torch.maximum(t1, t2).amin(0)) & (enter > 0) & (enter < best)
            best = torch.where(hit, enter, best)
            axis = torch.where(hit, ax.to(torch.uint8), axis)
        return best, axis

    def colour(self, p):
        chk = (torch.floor(p[0]) + torch.floor(p[1]) + torch.floor(2 * p[2])) % 2
        wave = torch.sin(p[None] * self.freq[:, :, None] + self.phase[:, :, None]).sum(1)
        return (0.55 * self.base[:, None] + 0.25 * chk + 0.07 * wave).clamp(0, 1)

    def returns(self, n, gen):
        """The first n LiDAR returns (points [3, n], face axes, ranges), scan by scan, each scan in
        beam and azimuth order with half of its returns dropped (more for a small map, so that it
        still comes from some eight scans)."""
        share = min(0.5, n / (8 * 30_000))
        el = torch.deg2rad(torch.linspace(-16, 15, 32, device=DEV))
        az = torch.deg2rad(torch.arange(0, 360, 0.2, device=DEV))
        parts, got = [], 0
        while got < n:
            s = torch.rand(min(64, max(1, int((n - got) / (20_000 * share)) + 1)), generator=gen, device=DEV)
            pos, _ = _path(self.scene, s.cpu().numpy().astype(np.float64))
            pos = torch.as_tensor(pos, dtype=torch.float32, device=DEV)
            rot = torch.rand(len(s), generator=gen, device=DEV) * math.radians(0.2)
            A = az[None, None, :] + rot[:, None, None]
            E = el[None, :, None].expand(len(s), -1, len(az))
            d = torch.stack([E.cos() * A.cos(), E.cos() * A.sin(), E.sin().expand(-1, -1, len(az))]).reshape(3, -1)
            o = pos.T[:, :, None].expand(-1, -1, 32 * len(az)).reshape(3, -1)
            r, ax = self.cast(o, d)
            keep = (r > 0.1) & (r < FAR) & (torch.rand(r.shape, generator=gen, device=DEV) < share)
            parts.append((o[:, keep] + r[keep] * d[:, keep], ax[keep], r[keep]))
            got += int(keep.sum())
        p, ax, r = (torch.cat(x, -1)[..., :n] for x in zip(*parts))
        return p, ax, r

    def image(self, cam):
        """Target colour [3, H, W] and camera-frame depth [H, W] (0: no return) of one camera."""
        W, H = cam["width"], cam["height"]
        R = torch.as_tensor(cam["R"], dtype=torch.float32, device=DEV)
        o = -(R.T @ torch.as_tensor(cam["t"], dtype=torch.float32, device=DEV))
        y, x = torch.meshgrid(torch.arange(H, device=DEV) + 0.5, torch.arange(W, device=DEV) + 0.5, indexing="ij")
        dc = torch.stack([(x - cam["cx"]) / cam["fx"], (y - cam["cy"]) / cam["fy"], torch.ones_like(x)]).reshape(3, -1)
        d = R.T @ dc
        z, _ = self.cast(o[:, None].expand_as(d), d)
        hit = z < FAR
        p = o[:, None] + torch.where(hit, z, 0) * d
        sky = torch.tensor([0.55, 0.65, 0.8], device=DEV)[:, None]
        return torch.where(hit, self.colour(p), sky).reshape(3, H, W), torch.where(hit, z, 0).reshape(H, W)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _gaussians(world, n, sh, gen):
    """Map planes [11 + 3K, n]: one Gaussian per return, flat along the surface."""
    p, ax, r = world.returns(n, gen)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=DEV)

    q = torch.zeros(4, n, device=DEV)
    q[0] = 1.0
    s2 = math.sqrt(0.5)
    for axis, quat in ((0, (s2, 0, s2, 0)), (1, (s2, -s2, 0, 0))):
        q = torch.where(ax == axis, torch.tensor(quat, device=DEV)[:, None], q)
    q = q + 0.05 * normal(4, n)
    tang = torch.log(torch.clamp(r * math.radians(0.4), min=0.01))
    out = [p + 0.01 * normal(3, n), tang + 0.2 * normal(2, n), math.log(0.01) + 0.2 * normal(1, n),
           q / q.norm(dim=0), normal(1, n), (world.colour(p) - 0.5) / Y00 + 0.05 * normal(3, n)]
    if sh:
        out.append(0.1 * normal(3 * (sh + 1) ** 2 - 3, n))
    return torch.cat(out).contiguous()


def _look(W, H, pos, heading, pitch=math.radians(5.0)):
    f = np.array([math.cos(heading) * math.cos(pitch), math.sin(heading) * math.cos(pitch), -math.sin(pitch)])
    r = np.cross(f, [0.0, 0.0, 1.0])
    r /= np.linalg.norm(r)
    R = np.stack([r, np.cross(f, r), f])
    return dict(width=W, height=H, fx=0.7 * W, fy=0.7 * W, cx=W / 2, cy=H / 2, R=R, t=-R @ pos)


def _cameras(scene, sizes, seed):
    """Keyframes at trajectory poses: half recent (the last tenth of the drive), half history."""
    rs = np.random.RandomState((seed + 7) % (1 << 31))
    out = []
    for k, (W, H) in enumerate(sizes):
        s = rs.uniform(0.9, 1.0) if k % 2 else rs.uniform(0.0, 0.9)
        if scene == "line":
            s *= 0.8                                            # something left to look at
        pos, head = _path(scene, np.array([s]))
        out.append(_look(W, H, pos[0], head[0]))
    return out


def _problem(case, seed):
    """Map planes, keyframes, packed target colour and depth."""
    gen, sizes = _gen(seed), _sizes(case)
    n, sh = case["n"], case["sh"]
    if case["scene"] == "box":        # a bounded volume before a camera at the origin
        lo, hi = torch.tensor([[-3.0, -3, 2], [3, 3, 10]], device=DEV)[:, :, None]

        def normal(*shape):
            return torch.randn(*shape, generator=gen, device=DEV)

        q = normal(4, n)
        planes = torch.cat([lo + (hi - lo) * torch.rand(3, n, generator=gen, device=DEV), -3 + 0.5 * normal(3, n),
                            q / q.norm(dim=0), normal(1, n), (torch.rand(3, n, generator=gen, device=DEV) - 0.5) / Y00,
                            0.1 * normal(3 * (sh + 1) ** 2 - 3, n)]).contiguous()
        cams = [dict(width=W, height=H, fx=0.9375 * W, fy=0.9375 * W, cx=W / 2, cy=H / 2, R=np.eye(3), t=np.zeros(3))
                for W, H in sizes]
        P = sum(w * h for w, h in sizes)
        return planes, cams, torch.rand(3 * P, generator=gen, device=DEV), 2 + 8 * torch.rand(P, generator=gen, device=DEV)
    world = _World(case["scene"], seed)
    planes = _gaussians(world, n, sh, gen)
    cams = _cameras(case["scene"], sizes, seed)
    images = [world.image(c) for c in cams]
    return planes, cams, torch.cat([i[0].reshape(-1) for i in images]), torch.cat([i[1].reshape(-1) for i in images])


def _max_pairs(case):
    return (1 << 21) + (3 if case["tile"] == 16 else 10) * case["n"] * len(_sizes(case))


def _moments(planes, pixels, gen):
    """Adam moments of a map some iterations into its optimisation."""
    s = 3.0 / pixels
    m = s * torch.randn(planes.shape, generator=gen, device=DEV)
    return m, s * s * (0.25 + torch.rand(planes.shape, generator=gen, device=DEV))


def _masks(case, pixels, seed):
    """(caller's mask of a step or None, rows that may change or None)"""
    gen = _gen(seed + 3)
    mask = (torch.rand(pixels, generator=gen, device=DEV) < 0.9).to(torch.uint8) if case["objective"] == "masked" else None
    upd = (torch.arange(case["n"], device=DEV) >= case["n"] // 2).to(torch.uint8) if case["mode"] == "parallel" else None
    return mask, upd


def _opts(case):
    extra = dict(lambda_ssim=0.2, mask_erode=2) if case.get("objective") == "ssim" else {}
    return gs.default_opts(tile=case["tile"], chunk=case["chunk"], **extra)


def _twists(V, seed):
    rs = np.random.RandomState((seed + 11) % (1 << 31))
    return torch.tensor(rs.normal(0, 0.01, (V, 6)), dtype=torch.float32)


# -- the passes --------------------------------------------------------------------------------

def _prepare_step(case, seed):
    planes, cams, trgb, tdep = _problem(case, seed)
    mode, P = case["mode"], tdep.numel()
    mask, upd = _masks(case, P, seed)
    s = dict(case=case, kept=planes.clone(), cams=cams, trgb=trgb, tdep=tdep, mask=mask, upd=upd)
    if mode == "parallel":
        s["par"] = gs.ViewParallelStep(planes, case["sh"], cams, _opts(case), max_pairs=_max_pairs(case))
        step = s["par"].step
    else:
        step = gs.MappingStep(planes, case["sh"], cams, _opts(case), max_pairs=_max_pairs(case))
    s["step"] = step
    if mode != "grads":
        m, v = _moments(planes, P, _gen(seed + 5))
        step.m.copy_(m)
        step.v.copy_(v)
    if mode == "graph":
        step.capture(trgb, tdep, mask)
    if mode == "host":
        host = (trgb.cpu().pin_memory(), tdep.cpu().pin_memory(), None if mask is None else mask.cpu().pin_memory(),
                torch.zeros(len(cams) + 1).pin_memory())
        step.capture(torch.empty_like(trgb), torch.empty_like(tdep), None if mask is None else torch.empty_like(mask),
                     host=host)
    return s


def _run_step(s):
    mode, step = s["case"]["mode"], s["step"]
    if mode == "grads":
        step.grads.zero_()
        r = step(s["trgb"], s["tdep"], s["mask"], optimize=False, with_twist=True)
        return dict(loss=r.loss, rgb=r.rgb, depth=r.depth, grads=step.grads, twist=step.twist)
    step.planes.copy_(s["kept"])
    if mode == "parallel":
        loss = s["par"](s["trgb"], s["tdep"], s["mask"], s["upd"])
        return dict(loss=loss, rgb=step.rgb, depth=step.depth, planes=step.planes, m=step.m, v=step.v,
                    twist=s["par"].twist)
    if mode == "eager":
        step.set_cameras(s["cams"])
        r = step(s["trgb"], s["tdep"], s["mask"])
    else:
        r = step.replay()
    return dict(loss=r.loss, rgb=r.rgb, depth=r.depth, planes=step.planes, m=step.m, v=step.v)


def _prepare_autograd(case, seed):
    planes, cams, _, _ = _problem(case, seed)
    gen = _gen(seed + 9)
    P = sum(w * h for w, h in _sizes(case))
    r = gs.Renderer(case["n"], cams, case["sh"], _opts(case), max_pairs=_max_pairs(case))
    return dict(case=case, r=r, planes=planes.requires_grad_(True), twist=_twists(len(cams), seed).requires_grad_(True),
                w_rgb=torch.randn(3 * P, generator=gen, device=DEV), w_depth=0.1 * torch.randn(P, generator=gen, device=DEV))


def _run_autograd(s):
    rgb, depth, T = s["r"](s["planes"], s["twist"])
    g, gt = torch.autograd.grad([rgb, depth], [s["planes"], s["twist"]], [s["w_rgb"], s["w_depth"]])
    return dict(rgb=rgb.detach(), depth=depth.detach(), T=T, grads=g, twist=gt)


def _prepare_render(case, seed):
    planes, cams, _, _ = _problem(case, seed)
    ws = gs.Workspace(case["n"], cams, _opts(case), _max_pairs(case))
    P = ws.layout.total_pixels
    return dict(case=case, planes=planes, ws=ws, rgb=torch.empty(3 * P, device=DEV), depth=torch.empty(P, device=DEV),
                T=torch.empty(P, device=DEV))


def _run_render(s):
    ws = s["ws"]
    ws.project(s["planes"], s["case"]["sh"])
    ws.bin_sort()
    ws.render_fwd(s["rgb"], s["depth"], s["T"])
    return dict(rgb=s["rgb"], depth=s["depth"], T=s["T"])


def _mlp_weights(seed):
    rs = np.random.RandomState((seed + 13) % (1 << 31))
    Ws = [rs.normal(0, math.sqrt(2.0 / i), (o, i)) for o, i in learned.LAYERS]
    Ws[-1] *= 0.1
    return Ws, [0.02 * rs.normal(0, 1, o) for o, _ in learned.LAYERS]


def _prepare_init(case, seed):
    gen, world = _gen(seed), _World("line", seed)
    p, _, _ = world.returns(case["n"], gen)
    col = world.colour(p)
    p = (p + 0.01 * torch.randn(p.shape, generator=gen, device=DEV)).contiguous()
    frames = _cameras("line", [(320, 240)] * case["frames"], seed)
    return dict(case=case, points=p, colours=col.contiguous(), frames=frames, mlp=learned.MLP(*learned.pack_params(*_mlp_weights(seed))))


def _run_init(s):
    pca = learned.voxel_pca(s["points"], s["colours"], s["frames"])
    y = s["mlp"].infer(pca["x"])
    planes, branch, beta = learned.cascade(s["points"], s["colours"], pca, float(s["frames"][0]["fx"]), y,
                                           sh_degree=s["case"]["sh"])
    return dict(planes=planes, branch=branch, beta=beta, y=y, **pca)


def _rotations(q):
    """Rotation matrices [n, 3, 3] of quaternions q [4, n] (w, x, y, z) of any length."""
    w, x, y, z = q / q.norm(dim=0)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z), 1 - 2 * (x * x + z * z),
                        2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _mlp_batch(n, seed):
    """Features as the voxel fit makes them (log variances, a rotation, colour, log footprint) and
    small residual targets."""
    gen = _gen(seed)
    x = torch.randn(n, 16, generator=gen, device=DEV)
    x[:, 0:3] = (-7 + 1.5 * x[:, 0:3]).sort(dim=1).values
    x[:, 3:12] = _rotations(x[:, 3:7].T).reshape(n, 9)
    x[:, 12:15] = torch.rand(n, 3, generator=gen, device=DEV)
    x[:, 15] = -3.5 + 0.5 * x[:, 15]
    y = torch.zeros(n, 16, device=DEV)
    y[:, :11] = 0.2 * torch.randn(n, 11, generator=gen, device=DEV)
    return x.contiguous(), y


def _prepare_mlp_train(case, seed):
    mlp = learned.MLP(*learned.pack_params(*_mlp_weights(seed)))
    gen = _gen(seed + 1)                                    # a hundred steps into its training
    mlp.t = 100
    mlp.m.copy_(1e-3 * torch.randn(mlp.m.shape, generator=gen, device=DEV))
    mlp.v.copy_(1e-6 * (0.25 + torch.rand(mlp.v.shape, generator=gen, device=DEV)))
    x, y = _mlp_batch(case["n"], seed)
    return dict(case=case, mlp=mlp, x=x, y=y)


def _run_mlp_train(s):
    mlp = s["mlp"]
    loss = mlp.train_step(s["x"], s["y"])
    return dict(loss=loss, w=mlp.w, b=mlp.b, m=mlp.m, v=mlp.v)


def _occupied(means, new, radius=0.05):
    """Whether a mean lies within `radius` of each new point (single-precision distances), from 5 cm
    cells and the points of the 27 cells around each new point."""
    side = 1.01 * radius

    def key(c):
        return (c[0] * (1 << 42) + c[1] * (1 << 21)) + c[2]

    ks, order = torch.sort(key(torch.floor(means.double() / side).long()))
    cq = torch.floor(new.double() / side).long()
    near = torch.zeros(new.shape[1], dtype=torch.bool, device=DEV)
    r2 = float(np.float32(radius) * np.float32(radius))
    for off in range(27):
        kq = key(cq + torch.tensor([off // 9 - 1, off // 3 % 3 - 1, off % 3 - 1], device=DEV)[:, None])
        lo, hi = torch.searchsorted(ks, kq), torch.searchsorted(ks, kq, right=True)
        for j in range(int((hi - lo).max())):
            at = torch.nonzero((lo + j < hi) & ~near).squeeze(1)
            if not len(at):
                break
            d = new[:, at] - means[:, order[lo[at] + j]]
            near[at] = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2] < r2
    return near


def _prepare_map_update(case, seed):
    """A map with 2% of faded rows (the removal ratio caps how many go) and new Gaussians of a revisited
    region, half of which the map already holds."""
    gen, world = _gen(seed), _World("loop", seed)
    n, k, sh = case["n"], case["new"], case["sh"]
    planes = _gaussians(world, n, sh, gen)
    planes[10] -= 10.0 * (torch.rand(n, generator=gen, device=DEV) < 0.02)
    new = planes[:, torch.randint(0, n, (3 * k,), generator=gen, device=DEV)].contiguous()
    new[0:3] += 0.1 * torch.randn(3, 3 * k, generator=gen, device=DEV)
    near = _occupied(planes[0:3], new[0:3])
    known, fresh = torch.nonzero(near).squeeze(1)[:k // 2], torch.nonzero(~near).squeeze(1)[:k - k // 2]
    short = torch.nonzero(near).squeeze(1)[k // 2:][: k - k // 2 - len(fresh)]
    new[0, short] += 500.0                                  # where the region is too dense: beyond it
    rows = torch.cat([known, fresh, short])
    near[short] = False
    spare = torch.nonzero(~near).squeeze(1)[k - k // 2:][: k - len(rows)]
    new[0:3, spare] = planes[0:3, : len(spare)] + 0.01      # too sparse: right beside its first rows
    new = new[:, torch.cat([rows, spare]).sort().values].contiguous()
    m, v = _moments(planes, 6_000_000, gen)
    tags = torch.randint(0, 8, (n,), generator=gen, device=DEV, dtype=torch.int32)
    return dict(case=case, planes=planes, m=m, v=v, new=new, tags=tags, new_tags=torch.full((k,), 8, dtype=torch.int32, device=DEV),
                scratch=gs.map_update_scratch(n, k))


def _run_map_update(s):
    sh = s["case"]["sh"]
    keep, kept = gs.prune_plan(s["planes"], sh, scratch=s["scratch"])
    accept, taken = gs.dedup_plan(s["planes"], sh, s["new"][0:3], scratch=s["scratch"])
    planes, m, v, tags = gs.map_update(s["planes"], s["m"], s["v"], sh, keep, s["new"], accept, s["tags"], s["new_tags"],
                                       scratch=s["scratch"])
    return dict(keep=keep, kept=kept, accept=accept, taken=taken, planes=planes, m=m, v=v, tags=tags)


def _rigid(xi):
    X = np.zeros((4, 4))
    X[:3, :3] = [[0, -xi[5], xi[4]], [xi[5], 0, -xi[3]], [-xi[4], xi[3], 0]]
    X[:3, 3] = xi[:3]
    return torch.linalg.matrix_exp(torch.tensor(X)).numpy()


def _prepare_gicp(case, seed):
    """A map, 4 query views around a loop frame, and a revisit: Gaussians of the same surfaces, a few
    centimetres and less than a degree off."""
    gen, world = _gen(seed), _World("loop", seed)
    planes = _gaussians(world, case["n"], 0, gen)
    rs = np.random.RandomState((seed + 17) % (1 << 31))
    s0 = rs.uniform(0, 0.95)
    views = []
    for ds in (0.0, 0.01, 0.02, 0.03):
        pos, head = _path("loop", np.array([s0 + ds]))
        views.append(_look(640, 480, pos[0], head[0]))
    c = torch.as_tensor(_path("loop", np.array([s0 + 0.02]))[0][0], dtype=torch.float32, device=DEV)
    near = (planes[0:3] - c[:, None]).norm(dim=0) < 20.0
    rows = torch.nonzero(near).squeeze(1)
    rows = rows[torch.randperm(len(rows), generator=gen, device=DEV)[: case["src"]]].sort().values
    T = _rigid(rs.uniform(-1, 1, 6) * np.array([0.05, 0.05, 0.02, 0.004, 0.004, 0.006]))
    src = planes[:, rows].contiguous()
    R, t = (torch.as_tensor(a, dtype=torch.float32, device=DEV) for a in (T[:3, :3], T[:3, 3:]))
    src[0:3] = R @ (src[0:3] + 0.003 * torch.randn(3, len(rows), generator=gen, device=DEV)) + t
    return dict(case=case, planes=planes, views=views, src=src, scratch=gs.gicp_scratch(case["n"]))


def _run_gicp(s):
    flag, count = gs.gicp_target_set(s["planes"], 0, s["views"], scratch=s["scratch"])
    T, res = gs.gicp_register(s["src"], None, s["planes"], flag, 0, scratch=s["scratch"])
    return dict(flag=flag, count=count, T=T, cost=float(res.cost), n_corr=int(res.n_corr), iters=int(res.iters))


_KINDS = dict(step=(_prepare_step, _run_step), autograd=(_prepare_autograd, _run_autograd),
              render=(_prepare_render, _run_render), init=(_prepare_init, _run_init),
              mlp_train=(_prepare_mlp_train, _run_mlp_train), map_update=(_prepare_map_update, _run_map_update),
              gicp=(_prepare_gicp, _run_gicp))


def prepare(case, seed):
    state = _KINDS[case["kind"]][0](case, seed)
    state["run"] = _KINDS[case["kind"]][1]
    return state


def run(state):
    return state["run"](state)


def work(case):
    kind, n = case["kind"], case["n"]
    if kind in ("step", "autograd", "render"):
        P, V = sum(w * h for w, h in _sizes(case)), len(_sizes(case))
        rows, evals = 11 + 3 * (case["sh"] + 1) ** 2, EVALS * P
        seen = n if case["scene"] == "box" else min(n, SEEN * n * V / 8)
        b = 44 * n + 4 * (rows - 11) * seen + 16 * P                 # the map in, images out
        if kind == "render":
            return dict(bytes=b + 4 * P, flops=evals * OPS_FWD)
        b += 16 * P                                                  # targets or upstream gradients in
        if kind == "autograd" or case["mode"] == "grads":
            return dict(bytes=b + 4 * rows * seen, flops=evals * (OPS_FWD + OPS_BWD))
        half = 0.5 if case["mode"] == "parallel" else 1.0
        ssim = 300 * P if case["objective"] == "ssim" else 0
        # the seen rows' parameters out, moments in and out; the kept map back into place
        return dict(bytes=b + 20 * rows * seen * half + 8 * rows * n, flops=evals * (OPS_FWD + OPS_BWD) + ssim)
    if kind == "init":
        # points and colours in, features, fits, network outputs and the planes out
        return dict(bytes=n * (24 + 2 * 64 + 12 + 16 + 4 + 3 + 4 + 4 * (11 + 3 * (case["sh"] + 1) ** 2)), flops=n * 2 * 36864)
    if kind == "mlp_train":
        return dict(bytes=n * 128 + 37264 * 28, flops=n * 6 * 36864)
    if kind == "map_update":
        rows, k = 11 + 3 * (case["sh"] + 1) ** 2, case["new"]
        return dict(bytes=24 * rows * n + 16 * rows * k + 20 * n, flops=10 * n)
    # the map's means against 4 views; 25 iterations over the pairs of Gaussians (40 B each)
    return dict(bytes=13 * n + 25 * 80 * case["src"], flops=n * 4 * 30 + 25 * case["src"] * 400)


# -- the same results in 64 bits, from plain torch ----------------------------------------------

NEAR, DILATION, A_MIN, A_MAX, T_MIN, CLAMP = 0.2, 0.3, 1.0 / 255.0, 0.99, 1e-4, 1.3


def _basis(deg, d):
    x, y, z = d
    Y = [torch.full_like(x, Y00)]
    if deg >= 1:
        c = math.sqrt(3 / (4 * math.pi))
        Y += [-c * y, c * z, -c * x]
    if deg >= 2:
        a, b, e = math.sqrt(15 / (4 * math.pi)), math.sqrt(5 / (16 * math.pi)), math.sqrt(15 / (16 * math.pi))
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, e * (x * x - y * y)]
    if deg >= 3:
        a, b, c = math.sqrt(35 / (32 * math.pi)), math.sqrt(105 / (4 * math.pi)), math.sqrt(21 / (32 * math.pi))
        e, f = math.sqrt(7 / (16 * math.pi)), math.sqrt(105 / (16 * math.pi))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              e * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y), f * z * (x * x - y * y),
              -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y)


def _pose(cam, twist):
    """R, t (as the single-precision camera record holds them), moved by Exp(twist) on the left."""
    R = torch.as_tensor(np.asarray(cam["R"], np.float32).astype(np.float64), device=DEV)
    t = torch.as_tensor(np.asarray(cam["t"], np.float32).astype(np.float64), device=DEV)
    o = torch.zeros((), dtype=torch.float64, device=DEV)
    a, b, c = twist[3], twist[4], twist[5]
    X = torch.stack([torch.stack([o, -c, b, twist[0]]), torch.stack([c, o, -a, twist[1]]),
                     torch.stack([-b, a, o, twist[2]]), torch.stack([o, o, o, o])])
    E = torch.linalg.matrix_exp(X)
    return E[:3, :3] @ R, E[:3, :3] @ t + E[:3, 3]


def _project64(p, deg, cam, twist):
    """(u, v, z, conic a b c, opacity, r, g, b) [10, n] and the 2-D variances [2, n]."""
    R, t = _pose(cam, twist)
    pc = R @ p[0:3] + t[:, None]
    z = pc[2]
    xz, yz = pc[0] / z, pc[1] / z
    lx, ly = CLAMP * 0.5 * cam["width"] / cam["fx"], CLAMP * 0.5 * cam["height"] / cam["fy"]
    q = p[6:10] / p[6:10].norm(dim=0)
    w, x, y, k = q
    Q = torch.stack([torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y)]),
                     torch.stack([2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x)]),
                     torch.stack([2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)])])
    M = torch.einsum("ij,jkn->ikn", R, Q * torch.exp(p[3:6])[None])
    jx = (M[0] - M[2] * xz.clamp(-lx, lx)) * (cam["fx"] / z)
    jy = (M[1] - M[2] * yz.clamp(-ly, ly)) * (cam["fy"] / z)
    A, B, D = (jx * jx).sum(0) + DILATION, (jx * jy).sum(0), (jy * jy).sum(0) + DILATION
    det = A * D - B * B
    d = p[0:3] + (R.T @ t)[:, None]
    Y = _basis(deg, d / d.norm(dim=0))
    rgb = (torch.einsum("kn,kcn->cn", Y, p[11:].reshape(len(Y), 3, p.shape[1])) + 0.5).clamp(min=0)
    rec = torch.stack([cam["fx"] * xz + cam["cx"], cam["fy"] * yz + cam["cy"], z, D / det, -B / det, A / det,
                       torch.sigmoid(p[10]), *rgb])
    return rec, torch.stack([A, D])


def _depth_key(p, cam, twist):
    """The compositing order is defined on a single-precision depth (products and sums fused) under
    the single-precision pose."""
    R, t = (a.float().double() for a in _pose(cam, twist))
    z = (p[0] * R[2, 0]).float().double()
    z = (p[1] * R[2, 1] + z).float().double()
    z = (p[2] * R[2, 2] + z).float()
    return z + t[2].float()


def _blend64(r, px, py):
    """Colour [3, m], depth [m] and final transmittance [m] of pixels from records r [10, k] in order."""
    dx, dy = px[None] - r[0][:, None], py[None] - r[1][:, None]
    e = -0.5 * (r[3][:, None] * dx * dx + 2 * r[4][:, None] * dx * dy + r[5][:, None] * dy * dy)
    a = (r[6][:, None] * torch.exp(e)).clamp(max=A_MAX)
    a = torch.where(a >= A_MIN, a, 0.0)
    logT = torch.cumsum(torch.log1p(-a), 0)
    T = torch.exp(logT)
    kept = T >= T_MIN
    w = a * torch.exp(logT - torch.log1p(-a)) * kept
    return r[7:10] @ w, r[2] @ w, torch.where(kept, T, 1.0).amin(0)


class _Splat64:
    """The renderer and its adjoint for one batch of views."""

    def __init__(self, planes, deg, cams, twists, tile):
        self.p, self.deg, self.cams, self.tw = planes.double(), deg, cams, twists.double().to(DEV)
        self.views, self.seen = [], torch.zeros(planes.shape[1], dtype=torch.bool, device=DEV)
        for cam, tw in zip(cams, self.tw):
            with torch.no_grad():
                z = _depth_key(self.p, cam, tw)
                rows = torch.nonzero((z > NEAR) & (torch.sigmoid(self.p[10]) >= A_MIN)).squeeze(1)
                rec, var = _project64(self.p[:, rows], deg, cam, tw)
                tau = 2 * torch.log(rec[6] / A_MIN)
                rx, ry = torch.ceil((tau * var[0]).sqrt()), torch.ceil((tau * var[1]).sqrt())
                W, H = cam["width"], cam["height"]
                ok = ((rec[0] + rx >= 0) & (rec[1] + ry >= 0) & (torch.floor((rec[0] - rx) / tile) < -(-W // tile)) &
                      (torch.floor((rec[1] - ry) / tile) < -(-H // tile)))
                order = torch.sort(z[rows[ok]], stable=True).indices
                rows = rows[ok][order]
                self.seen[rows] = True
                self.views.append((rows, rec[:, ok][:, order], rx[ok][order], ry[ok][order]))

    def _blocks(self, v, size=32):
        rows, rec, rx, ry = self.views[v]
        W, H = self.cams[v]["width"], self.cams[v]["height"]
        for y0 in range(0, H, size):
            y1 = min(H, y0 + size)
            band = torch.nonzero((rec[1] + ry >= y0) & (rec[1] - ry <= y1)).squeeze(1)
            bl, bh = rec[0][band] - rx[band], rec[0][band] + rx[band]
            for x0 in range(0, W, size):
                x1 = min(W, x0 + size)
                pick = band[(bh >= x0) & (bl <= x1)]
                py, px = torch.meshgrid(torch.arange(y0, y1, device=DEV) + 0.5, torch.arange(x0, x1, device=DEV) + 0.5, indexing="ij")
                yield pick, px.reshape(-1).double(), py.reshape(-1).double(), slice(y0, y1), slice(x0, x1)

    def images(self):
        out = []
        with torch.no_grad():
            for v, cam in enumerate(self.cams):
                C = torch.zeros(3, cam["height"], cam["width"], dtype=torch.float64, device=DEV)
                D, T = torch.zeros_like(C[0]), torch.ones_like(C[0])
                for pick, px, py, sy, sx in self._blocks(v):
                    if len(pick):
                        c, d, t = _blend64(self.views[v][1][:, pick], px, py)
                        shape = D[sy, sx].shape
                        C[:, sy, sx], D[sy, sx], T[sy, sx] = c.reshape(3, *shape), d.reshape(shape), t.reshape(shape)
                out.append((C, D, T))
        return out

    def backward(self, upstream):
        """Gradients [11 + 3K, n] and twists [V, 6] for per-view (dL/dC, dL/dD)."""
        grads, gtw = torch.zeros_like(self.p), torch.zeros_like(self.tw)
        for v, (gC, gD) in enumerate(upstream):
            rows, rec, _, _ = self.views[v]
            grec = torch.zeros_like(rec)
            for pick, px, py, sy, sx in self._blocks(v):
                if not len(pick):
                    continue
                r = rec[:, pick].detach().requires_grad_(True)
                c, d, _ = _blend64(r, px, py)
                (g,) = torch.autograd.grad([c, d], [r], [gC[:, sy, sx].reshape(3, -1), gD[sy, sx].reshape(-1)])
                grec[:, pick] += g
            p = self.p[:, rows].detach().requires_grad_(True)
            tw = self.tw[v].detach().requires_grad_(True)
            g, gt = torch.autograd.grad(_project64(p, self.deg, self.cams[v], tw)[0], [p, tw], grec)
            grads[:, rows] += g
            gtw[v] = gt
        return grads, gtw


def _pack(images):
    return [torch.cat([i[k].reshape(-1) for i in images]) for k in range(3)]


def _window(x):
    k = torch.exp(-((torch.arange(11, dtype=torch.float64) - 5) ** 2) / 4.5)
    k = (k / k.sum()).tolist()
    for dim in (-1, -2):
        n = x.shape[dim]
        pad = torch.nn.functional.pad(x, (5, 5, 0, 0) if dim == -1 else (0, 0, 5, 5))
        x = sum(w * pad.narrow(dim, i, n) for i, w in enumerate(k))
    return x


def _objective64(images, cams, trgb, tdep, mask, ssim):
    """Per-view losses and their mean, and the upstream gradients of the mean."""
    losses, up, at, V = [], [], 0, len(cams)
    for (C, D, T), cam in zip(images, cams):
        H, W = cam["height"], cam["width"]
        P = H * W
        x = trgb[3 * at:3 * (at + P)].double().reshape(3, H, W)
        y = tdep[at:at + P].double().reshape(H, W)
        M = torch.ones(H, W, dtype=torch.bool, device=DEV) if mask is None else mask[at:at + P].reshape(H, W) != 0
        if ssim:                                   # eroded support of the rendering, radius 2
            geo = torch.nn.functional.pad((1 - T >= 0.5), (2, 2, 2, 2))
            for dy in range(-2, 3):
                for dx in range(-2, 3):
                    if dx * dx + dy * dy <= 4:
                        M = M & geo[2 + dy:2 + dy + H, 2 + dx:2 + dx + W]
        C, D = C.detach().requires_grad_(True), D.detach().requires_grad_(True)
        nm, Md = M.sum().clamp(min=1), M & (y > 0)
        L = ((C - x).abs() * M).sum() / nm + 0.1 * ((D - y).abs() * Md).sum() / Md.sum().clamp(min=1)
        if ssim:
            a, b = C * M, x * M
            ma, mb = _window(a), _window(b)
            va, vb, vab = _window(a * a) - ma * ma, _window(b * b) - mb * mb, _window(a * b) - ma * mb
            S = (2 * ma * mb + 1e-4) * (2 * vab + 9e-4) / ((ma * ma + mb * mb + 1e-4) * (va + vb + 9e-4))
            L = L + 0.2 * (1 - (S * M).sum() / (3 * nm))
        gC, gD = torch.autograd.grad(L, [C, D])
        losses.append(L.detach())
        up.append((gC / V, gD / V))
        at += P
    losses = torch.stack(losses)
    return torch.cat([losses, losses.mean()[None]]), up


def _exact_step(case, seed):
    planes, cams, trgb, tdep = _problem(case, seed)
    P = tdep.numel()
    mask, upd = _masks(case, P, seed)
    S = _Splat64(planes, case["sh"], cams, torch.zeros(len(cams), 6), case["tile"])
    images = S.images()
    loss, up = _objective64(images, cams, trgb, tdep, mask, case["objective"] == "ssim")
    rgb, depth, _ = _pack(images)
    grads, twist = S.backward(up)
    if case["mode"] == "grads":
        return dict(loss=loss, rgb=rgb, depth=depth, grads=grads, twist=twist)
    m0, v0 = _moments(planes, P, _gen(seed + 5))
    b1, b2, eps = (float(np.float32(x)) for x in (0.9, 0.999, 1e-15))
    rows = S.seen if upd is None else S.seen & (upd != 0)
    m = torch.where(rows, b1 * m0.double() + (1 - b1) * grads, m0.double())
    v = torch.where(rows, b2 * v0.double() + (1 - b2) * grads * grads, v0.double())
    lr = torch.tensor([gs.LR_DEFAULT[k] for k in [0] * 3 + [1] * 3 + [2] * 4 + [3] + [4] * 3 + [5] * (planes.shape[0] - 14)],
                      dtype=torch.float32, device=DEV).double()[:, None]
    p = planes.double()
    p = torch.where(rows, p - lr * (m / (1 - b1)) / ((v / (1 - b2)).sqrt() + eps), p)
    out = dict(loss=loss, rgb=rgb, depth=depth, planes=p, m=m, v=v)
    if case["mode"] == "parallel":
        out["twist"] = twist
    return out


def _exact_autograd(case, seed):
    planes, cams, _, _ = _problem(case, seed)
    gen = _gen(seed + 9)
    P = sum(w * h for w, h in _sizes(case))
    w_rgb = torch.randn(3 * P, generator=gen, device=DEV).double()
    w_depth = (0.1 * torch.randn(P, generator=gen, device=DEV)).double()
    S = _Splat64(planes, case["sh"], cams, _twists(len(cams), seed), case["tile"])
    rgb, depth, T = _pack(S.images())
    up, at = [], 0
    for c in cams:
        H, W = c["height"], c["width"]
        up.append((w_rgb[3 * at:3 * (at + H * W)].reshape(3, H, W), w_depth[at:at + H * W].reshape(H, W)))
        at += H * W
    grads, twist = S.backward(up)
    return dict(rgb=rgb, depth=depth, T=T, grads=grads, twist=twist)


def _exact_render(case, seed):
    planes, cams, _, _ = _problem(case, seed)
    rgb, depth, T = _pack(_Splat64(planes, case["sh"], cams, torch.zeros(len(cams), 6), case["tile"]).images())
    return dict(rgb=rgb, depth=depth, T=T)


def _net64(x, Ws, bs):
    for k, (W, b) in enumerate(zip(Ws, bs)):
        x = x @ W.T + b
        if k < 3:
            x = torch.nn.functional.gelu(x)
    return x


def _weights64(seed):
    return [[torch.as_tensor(np.asarray(a, np.float32), device=DEV).double() for a in g] for g in _mlp_weights(seed)]


def _exact_init(case, seed):
    s = _prepare_init(case, seed)
    n, fx = case["n"], float(s["frames"][0]["fx"])
    p = s["points"].double()
    cell = torch.floor(s["points"] / 0.5).long()
    _, vox, cnt = torch.unique(cell[0] * (1 << 42) + cell[1] * (1 << 21) + cell[2], return_inverse=True, return_counts=True)
    N = cnt.double()
    mu = torch.zeros(3, len(cnt), dtype=torch.float64, device=DEV).index_add_(1, vox, p) / N
    d = p - mu[:, vox]
    Cov = torch.zeros(9, len(cnt), dtype=torch.float64, device=DEV).index_add_(1, vox, (d[:, None] * d[None]).reshape(9, n)) / N
    lam, V = torch.linalg.eigh(Cov.T.reshape(-1, 3, 3).cpu())
    lam, V = lam.to(DEV), V.to(DEV)
    big = V.abs().argmax(1, keepdim=True)
    V = V * torch.gather(V, 1, big).sign()
    V[:, :, 2] = torch.linalg.cross(V[:, :, 0], V[:, :, 1])
    has = cnt >= 5
    planar = lam[:, 0] < 2.5e-3
    k = torch.where(planar, 0, 2)
    classed = planar | (lam[:, 2] > 10 * lam[:, 0])
    lk = lam.gather(1, k[:, None])
    other = torch.arange(3, device=DEV)[None] != k[:, None]
    trace = 0.02 ** 2 * torch.where(other, (lam + lk) / (N[:, None] * (lk - lam) ** 2), 0.0).sum(1)
    top = lam[:, 2].clamp(min=1e-300)
    rel = has & classed & ((lam[:, 1] - lam[:, 0]) / top > 1e-6) & ((lam[:, 2] - lam[:, 1]) / top > 1e-6) & (trace < 1e-2)
    has, rel = has[vox], rel[vox]
    lam, V = lam[vox].clamp(min=1e-4), V[vox]
    depth, best = None, torch.full((n,), math.inf, dtype=torch.float64, device=DEV)
    for c in s["frames"]:
        R, t = _pose(c, torch.zeros(6, dtype=torch.float64, device=DEV))
        x, y, z = R @ p + t[:, None]
        depth = z if depth is None else depth
        u, v = c["fx"] * x / z + c["cx"], c["fy"] * y / z + c["cy"]
        best = torch.where((z > 0) & (u >= 0) & (u < c["width"]) & (v >= 0) & (v < c["height"]) & (z < best), z, best)
    inside = best.isfinite()
    depth = torch.where(inside, best, depth)
    foot = torch.log(depth.clamp(min=1e-6) / fx)
    x = torch.cat([lam.log(), V.reshape(n, 9), s["colours"].T.double(), foot[:, None]], 1) * has[:, None]
    y = _net64(x, *_weights64(seed))
    valid = has & inside & (y[:, 0:3].abs() < 3).all(1)
    beta = ((rel & ~valid).sum() / n).clamp(0.25, 1).double()
    # unit quaternion of V (w >= 0) through the eigenvector of the symmetric 4 x 4 form
    m = V
    K = torch.stack([m[:, 0, 0] - m[:, 1, 1] - m[:, 2, 2], m[:, 0, 1] + m[:, 1, 0], m[:, 0, 2] + m[:, 2, 0], m[:, 2, 1] - m[:, 1, 2],
                     m[:, 1, 1] - m[:, 0, 0] - m[:, 2, 2], m[:, 1, 2] + m[:, 2, 1], m[:, 0, 2] - m[:, 2, 0],
                     m[:, 2, 2] - m[:, 0, 0] - m[:, 1, 1], m[:, 1, 0] - m[:, 0, 1], m[:, 0, 0] + m[:, 1, 1] + m[:, 2, 2]], 1)
    B = K[:, [0, 1, 2, 3, 1, 4, 5, 6, 2, 5, 7, 8, 3, 6, 8, 9]].reshape(n, 4, 4)
    S = B + 3.0 * torch.eye(4, dtype=torch.float64, device=DEV)     # 4 q q^T, q = (x, y, z, w)
    q = S.gather(2, S.diagonal(dim1=1, dim2=2).argmax(1)[:, None, None].expand(-1, 4, 1)).squeeze(2)[:, [3, 0, 1, 2]]
    q = q / q.norm(dim=1, keepdim=True)
    q = torch.where(q[:, :1] < 0, -q, q)
    q = torch.where(has[:, None], q, torch.tensor([1.0, 0, 0, 0], dtype=torch.float64, device=DEV))
    spca = 0.5 * lam.log() * has[:, None]
    qm = q + y[:, 3:7]
    logit = math.log(0.1 / 0.9)
    a, b = valid[:, None], rel[:, None]
    ls = torch.where(a, spca + y[:, 0:3], torch.where(b, spca + beta.log(), foot[:, None]))
    qq = torch.where(a, qm / qm.norm(dim=1, keepdim=True), torch.where(b, q, torch.tensor([1.0, 0, 0, 0], dtype=torch.float64, device=DEV)))
    col = s["colours"].T.double() + torch.where(a, y[:, 8:11], 0.0)
    out = torch.zeros(11 + 3 * (case["sh"] + 1) ** 2, n, dtype=torch.float64, device=DEV)
    out[0:3], out[3:6], out[6:10], out[10], out[11:14] = p, ls.T, qq.T, logit + torch.where(valid, y[:, 7], 0.0), ((col - 0.5) / Y00).T
    # the fits of voxels without a feature are not defined: no value for s_pca and q_pca
    return dict(planes=out, branch=None, beta=beta[None], y=y, x=x, has_feature=None, reliable=None, s_pca=None, q_pca=None,
                depth=depth, inside=None)


def _exact_mlp_train(case, seed):
    s = _prepare_mlp_train(case, seed)
    Ws, bs = _weights64(seed)
    leaves = [a.requires_grad_(True) for a in Ws + bs]
    y = _net64(s["x"].double(), Ws, bs)
    loss = ((y - s["y"].double())[:, :11] ** 2).sum() / (case["n"] * 11)
    g = torch.autograd.grad(loss, leaves)
    g = torch.cat([a.reshape(-1) for a in g])
    p = torch.cat([a.detach().reshape(-1) for a in leaves])
    b1, b2, eps, lr = (float(np.float32(a)) for a in (0.9, 0.999, 1e-8, 1e-3))
    m = b1 * s["mlp"].m.double() + (1 - b1) * g
    v = b2 * s["mlp"].v.double() + (1 - b2) * g * g
    p = p - lr * (m / (1 - b1 ** 101)) / ((v / (1 - b2 ** 101)).sqrt() + eps)
    return dict(loss=loss.detach()[None], w=p[:36864], b=p[36864:], m=m, v=v)


def _exact_map_update(case, seed):
    s = _prepare_map_update(case, seed)
    n, k = case["n"], case["new"]
    logit = s["planes"][10]
    low = torch.nonzero(logit < float(np.float32(math.log(0.005 / 0.995)))).squeeze(1)
    gone = low[torch.sort(logit[low], stable=True).indices][: int(0.01 * n)]
    keep = torch.ones(n, dtype=torch.bool, device=DEV)
    keep[gone] = False
    new = s["new"][:, ~_occupied(s["planes"][0:3], s["new"][0:3])].double()
    return dict(keep=None, kept=None, accept=None, taken=None, tags=None,
                planes=torch.cat([s["planes"][:, keep].double(), new], 1),
                m=torch.cat([s["m"][:, keep].double(), torch.zeros_like(new)], 1),
                v=torch.cat([s["v"][:, keep].double(), torch.zeros_like(new)], 1))


def _planar64(p):
    R = _rotations(p[6:10].double())
    lam = torch.ones(p.shape[1], 3, dtype=torch.float64, device=DEV)
    lam.scatter_(1, p[3:6].argmin(0)[:, None], 1e-3)
    return (R * lam[:, None, :]) @ R.transpose(1, 2)


def _exact_gicp(case, seed):
    s = _prepare_gicp(case, seed)
    mean = s["planes"][0:3]
    flag = torch.zeros(case["n"], dtype=torch.bool, device=DEV)
    for c in s["views"]:
        R, t = np.asarray(c["R"], np.float32), np.asarray(c["t"], np.float32)
        pc = [(mean[0] * float(R[r, 0]) + mean[1] * float(R[r, 1])) + mean[2] * float(R[r, 2]) + float(t[r]) for r in range(3)]
        u, v = pc[0] * c["fx"] / pc[2] + c["cx"], pc[1] * c["fy"] / pc[2] + c["cy"]
        o = -(R.astype(np.float64).T @ t.astype(np.float64))
        d = mean - torch.as_tensor(o, dtype=torch.float32, device=DEV)[:, None]
        flag |= ((pc[2] > 0.2) & (u >= 0) & (u < c["width"]) & (v >= 0) & (v < c["height"]) &
                 ((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2] < 400.0))
    rows = torch.nonzero(flag).squeeze(1)
    tar, src = mean[:, rows], s["src"][0:3]
    ct, cs = _planar64(s["planes"][:, rows]), _planar64(s["src"])
    T = torch.eye(4, dtype=torch.float64)

    def pairs(T):
        R, t = T[:3, :3].float().to(DEV), T[:3, 3].float().to(DEV)
        q = torch.stack([(R[r, 0] * src[0] + R[r, 1] * src[1]) + R[r, 2] * src[2] + t[r] for r in range(3)])
        best, at = [], []
        for j in range(0, q.shape[1], 2048):
            d = [q[a, j:j + 2048, None] - tar[a, None] for a in range(3)]
            b, i = ((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]).min(1)
            best.append(b)
            at.append(i)
        best, at = torch.cat(best), torch.cat(at)
        ok = torch.nonzero(best < 1.0).squeeze(1)
        R, t = T[:3, :3].to(DEV), T[:3, 3].to(DEV)
        x = R @ src[:, ok].double() + t[:, None]
        r = (tar[:, at[ok]].double() - x).T
        a, b, c = (ct[at[ok]] + R @ cs[ok] @ R.T).unbind(1)       # inverse of the 3 x 3 rows
        W = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], 2)
        W = W / (a * torch.linalg.cross(b, c)).sum(1)[:, None, None]
        J = torch.zeros(len(ok), 3, 6, dtype=torch.float64, device=DEV)
        J[:, 0, 0] = J[:, 1, 1] = J[:, 2, 2] = -1
        J[:, 0, 4], J[:, 0, 5], J[:, 1, 3] = -x[2], x[1], x[2]
        J[:, 1, 5], J[:, 2, 3], J[:, 2, 4] = -x[0], -x[1], x[0]
        WJ = W @ J
        return (J.transpose(1, 2) @ WJ).sum(0).cpu(), (WJ * r[:, :, None]).sum((0, 1)).cpu(), float(((W @ r[:, :, None]).squeeze(2) * r).sum())

    for _ in range(30):
        H, g, _ = pairs(T)
        xi = -torch.linalg.solve(H, g)
        T = torch.as_tensor(_rigid(xi.numpy())) @ T
        if xi.norm() < 1e-7:
            break
    return dict(flag=None, count=None, T=T, cost=pairs(T)[2], n_corr=None, iters=None)


_EXACT = dict(step=_exact_step, autograd=_exact_autograd, render=_exact_render, init=_exact_init,
              mlp_train=_exact_mlp_train, map_update=_exact_map_update, gicp=_exact_gicp)


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)

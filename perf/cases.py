"""What is timed: the calls a user of the rasterizer makes, over the range of
sizes its configurations, tests and benchmark use.

Every case goes through the public entry points (``Renderer``, ``Frame``,
``render_differentiable``, ``render_multi``, ``rgb_loss``, ``BatchGraph``,
``sort_pairs``, ``Server``).  Scenes are drawn on the GPU from the case's
seed with the distributions of ``synth`` (the plain 2,000-Gaussian scene and
the urban street).  ``exact`` restates the whole map in float64 with plain
torch: projection, per-tile front-to-back blending with the documented
gates, and its gradient.
"""
import math

import numpy as np
import torch

from paper_2311_18561_gb300 import abi
from paper_2311_18561_gb300 import batch as B
from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import serve as SV
from paper_2311_18561_gb300 import synth

VGA, KITTI, HALF, FULL = "640x480", "1242x375", "960x640", "1920x1280"
# compositing configurations that the autotuner picks, and the default
TILES = ("16,16,1", "16,8,1", "16,16,2", "32,16,4", "16,32,4", "32,32,4")


def listed():
    return [
        # a preview of the plain configuration: the smallest render, all launches and latency
        dict(name="plain_view", kind="forward", scene="plain", n=2000, degree=0, views="160x120", tile="16,16,1"),
        # the same size through torch.autograd, as a first training script does it
        dict(name="plain_autograd", kind="autograd", scene="plain", n=2000, degree=3, views="160x120",
             tile="16,16,1"),
        # novel-view rendering of a street scene at the camera's full resolution, tuned tiles
        dict(name="urban_view", kind="forward", scene="urban", n=1_500_000, degree=3, views=FULL, tile="32,32,4"),
        # interactive viewing of two small scenes side by side, default tiles
        dict(name="two_scene_views", kind="multi", scene="urban", n=250_000, degree=1,
             views=" ".join([VGA, "641x479", VGA, "640x360"]), tile="16,16,1"),
        # the headline training step: forward + L1 + backward, captured once and replayed
        dict(name="urban_step", kind="graph", scene="urban", n=1_500_000, degree=3, views=FULL, tile="32,32,4"),
        # the training configuration at the KITTI geometry with the paper's loss, call by call
        dict(name="training_step", kind="step", scene="urban", n=1_000_000, degree=3, views=KITTI, tile="16,8,1"),
        # a batch of views of uneven size as one captured graph
        dict(name="batched_step", kind="graph", scene="urban", n=1_000_000, degree=3,
             views=" ".join([FULL, KITTI, HALF] * 4), tile="16,16,2"),
        # sky refinement, temporal smoothing and depth / opacity supervision at an odd size
        dict(name="sky_depth_step", kind="aux", scene="urban", n=300_000, degree=2, views="961x641", tile="16,16,1"),
        # velocity, staticness and 19-class semantic maps with their gradients
        dict(name="semantic_step", kind="features", scene="urban", n=200_000, degree=3, views=KITTI,
             tile="16,16,1"),
        # the photometric loss and its gradient on a full-resolution image
        dict(name="photometric_loss", kind="loss", height=1280, width=1920),
        # the public radix sort on full 32-bit keys
        dict(name="sort_8m", kind="sort", n=8_000_003, bits=32),
        # a burst of mixed requests to the render server over two resident scenes
        dict(name="serve_burst", kind="serve", scene="urban", n=500_000, degree=3, requests=24, tile="16,16,1"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo=64, hi=1920):
    w = _log_uniform(rng, lo, hi)
    return "%dx%d" % (w, max(48, min(1280, int(w / rng.choice((4 / 3, 1.5, 1.5, 3.3))))))


def draw(rng):
    kind = rng.choice(("forward", "forward", "autograd", "multi", "graph", "graph", "step", "step", "aux",
                       "features", "loss", "sort", "serve"))
    if kind == "loss":
        return dict(kind=kind, height=_log_uniform(rng, 48, 1280), width=_log_uniform(rng, 64, 1920))
    if kind == "sort":
        return dict(kind=kind, n=_log_uniform(rng, 1000, 16_000_000), bits=rng.choice((13, 31, 32)))
    c = dict(kind=kind, scene="urban", n=_log_uniform(rng, 20_000, 1_500_000), degree=rng.choice((0, 1, 2, 3, 3)),
             tile=rng.choice(TILES))
    if kind == "serve":
        return dict(c, n=min(c["n"], 500_000), requests=rng.randint(3, 24))
    if kind in ("autograd", "forward") and rng.random() < 0.5:  # small scenes
        return dict(c, scene="plain", n=_log_uniform(rng, 300, 20_000), views=_size(rng, 64, 640))
    n_views = rng.randint(2, 6) if kind in ("multi", "graph") else 1
    if n_views > 1:
        c["n"] = min(c["n"], 1_000_000)
    if kind == "features":
        c["n"] = min(c["n"], 300_000)
        return dict(c, views=_size(rng, 64, 1242))
    return dict(c, views=" ".join(_size(rng, 160) for _ in range(n_views)))


# --------------------------------------------------------------------------- inputs

def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=g.device) * (hi - lo) + lo


def _normal(g, mean, std, *shape):
    return torch.randn(*shape, generator=g, device=g.device) * std + mean


def _scene(which, n, degree, g):
    """``synth.make_plain_scene`` / ``make_urban_scene`` drawn on the GPU."""
    k = (degree + 1) ** 2
    if which == "plain":
        mu, vel = _uniform(g, -1.0, 1.0, n, 3), _normal(g, 0.0, 0.2, n, 3)
        beta, period = _uniform(g, 0.1, 2.0, n), _normal(g, 0.0, 0.3, n).exp()
        scale = _normal(g, -3.0, 0.5, n, 3).exp()
        sh = _normal(g, 0.0, 0.1, n, k, 3)
        sh[:, 0] = (_uniform(g, 0.0, 1.0, n, 3) - 0.5) * (2.0 * math.sqrt(math.pi))
    else:
        n_ground, n_facade = int(round(0.7 * n)), int(round(0.1 * n))
        n_static = n_ground + n_facade
        n_obj = n - n_static
        mu = torch.empty(n, 3, device="cuda")
        mu[:, 0] = _uniform(g, -100.0, 100.0, n)
        mu[:, 1] = _uniform(g, -30.0, 30.0, n)
        mu[:, 2] = _uniform(g, 0.0, 0.5, n)
        side = torch.where(_uniform(g, 0.0, 1.0, n_facade) < 0.5, -15.0, 15.0)
        mu[n_ground:n_static, 1] = side + _normal(g, 0.0, 0.3, n_facade)
        mu[n_ground:n_static, 2] = _uniform(g, 0.0, 20.0, n_facade)
        centre = torch.stack([_uniform(g, -100.0, 100.0, 300), _uniform(g, -12.0, 12.0, 300)], 1)
        cid = torch.randint(0, 300, (n_obj,), generator=g, device="cuda")
        mu[n_static:, :2] = centre[cid] + _normal(g, 0.0, 1.0, n_obj, 2)
        mu[n_static:, 2] = _uniform(g, 0.0, 3.0, n_obj)
        vel = torch.zeros(n, 3, device="cuda")
        ang, spd = _uniform(g, 0.0, 2 * math.pi, n_static), _uniform(g, 0.0, 0.25, n_static)
        vel[:n_static, 0], vel[:n_static, 1] = spd * ang.cos(), spd * ang.sin()
        ang, spd = _uniform(g, 0.0, 2 * math.pi, 300), _uniform(g, 0.0, 75.0, 300)
        vel[n_static:, 0], vel[n_static:, 1] = (spd * ang.cos())[cid], (spd * ang.sin())[cid]
        beta = _uniform(g, 5.0, 10.0, n)
        beta[n_static:] = _uniform(g, 0.05, 0.5, n_obj)
        period = _normal(g, 0.0, 0.5, n).exp()
        scale = _normal(g, -2.0, 0.5, n, 3).exp()
        sh = _normal(g, 0.0, 0.1, n, k, 3)
    return dict(mu=mu, vel=vel, tau=_uniform(g, 0.0, 1.0, n), beta=beta, period=period, scale=scale,
                quat=_normal(g, 0.0, 1.0, n, 4), opacity=torch.sigmoid(_normal(g, 0.0, 1.0, n)), sh=sh)


def _sizes(case):
    return [tuple(int(x) for x in v.split("x")) for v in case["views"].split()]


def _cams(case, rng, jitter_from=None):
    cams = []
    for w, h in _sizes(case):
        if case["scene"] == "plain":
            cams.append(synth.plain_camera(w, h, t=float(rng.uniform(0.3, 0.7))))
        else:
            fx = 720.0 * w / 1242 if w > 2.5 * h else None
            cams.append(synth.street_camera(float(rng.uniform(0.2, 0.7)), w, h, fx=fx,
                                            lateral=float(rng.uniform(-2.0, 2.0))))
    if jitter_from is not None:
        for c in cams:
            c["dt"] = float(rng.uniform(-0.02, 0.02))
            c["sky_jitter"] = _uniform(jitter_from, -0.5, 0.5, 2, c["height"], c["width"])
    return cams


def _inputs(case, seed):
    """Everything drawn for a case: the same for ``prepare`` and ``exact``."""
    g, rng, kind = _gen(seed), np.random.default_rng(int(seed)), case["kind"]
    if kind == "loss":
        shape = (3, case["height"], case["width"])
        tgt = _uniform(g, 0.0, 1.0, *shape)
        return dict(target=tgt, pred=(tgt + _normal(g, 0.0, 0.1, *shape)).clamp(0.0, 1.0))
    if kind == "sort":
        n, bits = case["n"], case["bits"]
        keys = torch.randint(0, 1 << bits, (n,), generator=g, device="cuda")
        keys = torch.where(keys >= 1 << 31, keys - (1 << 32), keys).to(torch.int32)
        return dict(keys=keys, vals=torch.arange(n, device="cuda", dtype=torch.int32))
    if kind == "serve":
        scenes = [_scene("urban", m, case["degree"], g) for m in (case["n"], 2 * case["n"])]
        reqs = []
        for k in range(case["requests"]):
            w, h = synth.SERVE_RESOLUTIONS[k % len(synth.SERVE_RESOLUTIONS)]
            cam = synth.street_camera(float(rng.uniform(0.0, 1.0)), w, h, lateral=float(rng.uniform(-2.0, 2.0)))
            reqs.append((int(rng.integers(0, 2)), cam))
        return dict(scenes=scenes, reqs=reqs)
    cams = _cams(case, rng, g if kind == "aux" else None)
    if kind == "multi":
        return dict(scenes=[_scene(case["scene"], case["n"], case["degree"], g) for _ in range(2)], cams=cams)
    st = _scene(case["scene"], case["n"], case["degree"], g)
    d = dict(scene=st, cams=cams)
    if kind == "aux":
        st["sky"] = _uniform(g, 0.0, 1.0, 6, 256, 256, 3)
    if kind == "features":
        st["sem"] = torch.softmax(_normal(g, 0.0, 1.5, case["n"], 19), 1)
    if kind in ("graph", "step"):
        d["targets"] = [_uniform(g, 0.0, 1.0, 3, c["height"], c["width"]) for c in cams]
    if kind in ("autograd", "aux", "features"):
        c = cams[0]
        h, w = c["height"], c["width"]
        d["dl"] = dict(rgb=_normal(g, 0.0, 1.0 / (h * w), 3, h, w), depth=_normal(g, 0.0, 0.1 / (h * w), h, w),
                       alpha=_normal(g, 0.0, 1.0 / (h * w), h, w))
        if kind == "features":
            d["dl"]["feat"] = _normal(g, 0.0, 0.1 / (h * w), 23, h, w)
    return d


class _Serving:
    def __init__(self, d, tile):
        tw, th, px = tile
        self.server = SV.Server(tile=(tw, th), pixels_per_thread=px, memory_budget=3 << 30)
        self.ids = [self.server.add_scene(s) for s in d["scenes"]]
        self.reqs = d["reqs"]
        self.outs = [dict(rgb=torch.empty(3, c["height"], c["width"], device="cuda")) for _, c in self.reqs]


def prepare(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    s = dict(d, kind=kind, bits=case.get("bits"))
    if kind in ("loss", "sort"):
        s["r"] = R.Renderer()
        return s
    tw, th, px = (int(x) for x in case["tile"].split(","))
    if kind == "serve":
        s["serving"] = _Serving(d, (tw, th, px))
        return s
    if kind == "graph":
        s["graph"] = B.BatchGraph(d["scene"], d["cams"], targets=d["targets"], config=(tw, th, px))
        return s
    s["r"] = r = R.Renderer(tile=(tw, th), pixels_per_thread=px)
    feats = abi.FEAT_VBAR | abi.FEAT_RHO | abi.FEAT_SEM if kind == "features" else 0
    s["features"] = feats
    if kind == "autograd":
        s["params"] = {k: v.clone().requires_grad_(True) for k, v in d["scene"].items()}
        return s
    s["outs"] = r.alloc_images(d["cams"], features=feats, n_sem=19)
    if kind in ("step", "aux", "features"):
        s["frame"] = R.Frame()
        s["grads"] = {k: torch.empty_like(v) for k, v in d["scene"].items()}
    return s


# --------------------------------------------------------------------------- the calls

def run(s):
    kind = s["kind"]
    if kind == "forward":
        return s["r"].forward(s["scene"], s["cams"], outs=s["outs"])
    if kind == "multi":
        return R.render_multi(s["r"], [s["scenes"][v % 2] for v in range(len(s["cams"]))], s["cams"], outs=s["outs"])
    if kind == "autograd":
        rgb, depth, alpha = R.render_differentiable(s["params"], s["cams"][0], s["r"])
        dl = s["dl"]
        grads = torch.autograd.grad((rgb, depth, alpha), [s["params"][k] for k in R.PARAM_NAMES],
                                    (dl["rgb"], dl["depth"], dl["alpha"]))
        return dict(rgb=rgb, depth=depth, alpha=alpha, grads=dict(zip(R.PARAM_NAMES, grads)))
    if kind == "graph":
        g = s["graph"]
        g.replay()
        return dict(images=g.outs, losses=g.losses, grads=g.grads)
    if kind == "step":
        out = s["r"].forward(s["scene"], s["cams"], outs=s["outs"], frame=s["frame"])[0]
        loss, dl = R.rgb_loss(s["r"], out["rgb"], s["targets"][0])
        grads = s["r"].backward(s["scene"], s["cams"], s["frame"], [dict(rgb=dl)], grads=s["grads"])
        return dict(images=out, loss=loss, grads=grads)
    if kind in ("aux", "features"):
        out = s["r"].forward(s["scene"], s["cams"], outs=s["outs"], frame=s["frame"], features=s["features"])[0]
        grads = s["r"].backward(s["scene"], s["cams"], s["frame"], [s["dl"]], grads=s["grads"])
        return dict(images=out, grads=grads)
    if kind == "loss":
        loss, dl = R.rgb_loss(s["r"], s["pred"], s["target"])
        return dict(loss=loss, dl=dl)
    if kind == "sort":
        keys, vals = R.sort_pairs(s["r"], s["keys"].clone(), s["vals"].clone(), 0, s["bits"])
        return dict(keys=keys, vals=vals)
    sv = s["serving"]
    ids = [sv.server.submit(sv.ids[k], cam, out) for (k, cam), out in zip(sv.reqs, sv.outs)]
    for i in ids:
        sv.server.wait(i)
    for i in ids:
        sv.server.release(i)
    return [o["rgb"] for o in sv.outs]


def work(case):
    """Parameters and targets read once, images and gradients written once;
    arithmetic per Gaussian (time evaluation, projection, colour; about three
    times that in the adjoint) and per pixel at the 100 blended entries a
    street pixel takes before it saturates (14 operations each, 37 in the
    adjoint; 2 and 4 more per extra channel)."""
    kind = case["kind"]
    if kind == "loss":
        n = 3 * case["height"] * case["width"]
        return dict(bytes=12.0 * n, flops=207.0 * 2 * n)
    if kind == "sort":
        return dict(bytes=16.0 * case["n"], flops=0.0)
    params = 17 + 3 * (case["degree"] + 1) ** 2
    if kind == "serve":
        px = case["requests"] * sum(w * h for w, h in synth.SERVE_RESOLUTIONS) / 3.0
        n = 1.5 * case["n"] * case["requests"]
        return dict(bytes=4.0 * (params * n + 3 * px), flops=300.0 * n + 1400.0 * px)
    px = float(sum(w * h for w, h in _sizes(case)))
    scenes, views = (2 if kind == "multi" else 1), len(_sizes(case))
    n = float(case["n"])
    b, f = 4.0 * (params * n * scenes + 5 * px), 300.0 * n * views + 1400.0 * px
    if kind in ("graph", "step"):
        b, f = b + 4.0 * (params * n + 3 * px), f + 900.0 * n * views + 3700.0 * px
    if kind in ("autograd", "aux", "features"):
        b, f = b + 4.0 * (params * n + 5 * px), f + 900.0 * n + 3700.0 * px
    if kind == "features":
        b, f = b + 4.0 * (2 * 19 * n + 2 * 23 * px), f + 600.0 * 23 * px
    return dict(bytes=b, flops=f)


# --------------------------------------------------------------------------- float64

F64 = torch.float64


def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    pi = math.pi
    out = [torch.full_like(x, 0.5 * math.sqrt(1 / pi))]
    if degree >= 1:
        c = math.sqrt(3 / (4 * pi))
        out += [-c * y, c * z, -c * x]
    if degree >= 2:
        c, c0, c2 = 0.5 * math.sqrt(15 / pi), 0.25 * math.sqrt(5 / pi), 0.25 * math.sqrt(15 / pi)
        out += [c * x * y, -c * y * z, c0 * (2 * z * z - x * x - y * y), -c * x * z, c2 * (x * x - y * y)]
    if degree >= 3:
        c3, c2 = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi)
        c1, c0, ce = 0.25 * math.sqrt(21 / (2 * pi)), 0.25 * math.sqrt(7 / pi), 0.25 * math.sqrt(105 / pi)
        out += [-c3 * y * (3 * x * x - y * y), c2 * x * y * z, -c1 * y * (4 * z * z - x * x - y * y),
                c0 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c1 * x * (4 * z * z - x * x - y * y),
                ce * z * (x * x - y * y), -c3 * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _cam64(cam):
    f = lambda v: float(np.float32(v))  # noqa: E731  the library takes float32 cameras
    vm = torch.tensor(np.asarray(cam["viewmat"], np.float32).astype(np.float64), device="cuda")
    return dict(Rm=vm[:, :3], T=vm[:, 3], fx=f(cam["fx"]), fy=f(cam["fy"]), cx=f(cam["cx"]), cy=f(cam["cy"]),
                W=cam["width"], H=cam["height"], t=f(cam["t"]), zn=f(cam["z_near"]), dt=f(cam["dt"]),
                bg=torch.tensor(np.asarray(cam["bg"], np.float64), device="cuda"))


def _project64(P, C, degree, feats):
    """Screen-space terms of every Gaussian, and which of them can be seen."""
    delta = (C["t"] - C["dt"]) - P["tau"]
    vbw = torch.exp(-0.5 * P["beta"] / P["period"])
    amp = P["period"] * torch.sin(2 * math.pi * delta / P["period"]) / (2 * math.pi)
    if C["dt"] != 0.0:
        amp = amp + C["dt"] * vbw
    mut = P["mu"] + amp[:, None] * P["vel"]
    ot = P["opacity"] * torch.exp(-0.5 * delta ** 2 / P["beta"] ** 2)
    p = mut @ C["Rm"].T + C["T"]
    z = p[:, 2]
    seen = ((z > C["zn"]) & (ot >= 1 / 255)).nonzero()[:, 0]
    p, z, ot, mut = p[seen], z[seen], ot[seen], mut[seen]
    q = P["quat"][seen]
    w, x, y, zq = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + zq * zq), 2 * (x * y - w * zq), 2 * (x * zq + w * y),
                      2 * (x * y + w * zq), 1 - 2 * (x * x + zq * zq), 2 * (y * zq - w * x),
                      2 * (x * zq - w * y), 2 * (y * zq + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = Rq * P["scale"][seen][:, None, :]
    limx, limy = 1.3 * 0.5 * C["W"] / C["fx"], 1.3 * 0.5 * C["H"] / C["fy"]
    rx, ry = (p[:, 0] / z).clamp(-limx, limx), (p[:, 1] / z).clamp(-limy, limy)
    Rm = C["Rm"]
    T0 = (C["fx"] / z)[:, None] * Rm[0] - (C["fx"] * rx / z)[:, None] * Rm[2]
    T1 = (C["fy"] / z)[:, None] * Rm[1] - (C["fy"] * ry / z)[:, None] * Rm[2]
    U0, U1 = torch.einsum("nk,nkj->nj", T0, M), torch.einsum("nk,nkj->nj", T1, M)
    h = float(np.float32(0.3))
    A, Bc, Cc = (U0 * U0).sum(1) + h, (U0 * U1).sum(1), (U1 * U1).sum(1) + h
    det = A * Cc - Bc * Bc
    u, v = C["fx"] * p[:, 0] / z + C["cx"], C["fy"] * p[:, 1] / z + C["cy"]
    campos = -C["Rm"].T @ C["T"]
    d = mut - campos
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), degree)
    rgb = (torch.einsum("nk,nkc->nc", Y, P["sh"][seen]) + 0.5).clamp_min(0.0)
    terms = dict(u=u, v=v, a=Cc / det, b=-Bc / det, c=A / det, o=ot, z=z, rgb=rgb)
    if feats:
        terms["feat"] = torch.cat([P["vel"][seen] * vbw[seen][:, None],
                                   (P["beta"] / P["period"])[seen].clamp_max(2.0)[:, None], P["sem"][seen]], 1)
    with torch.no_grad():
        Q = (2 * torch.log(255 * ot)).clamp_min(0.0)
        box = torch.stack([u - torch.sqrt(Q * A) - 1, u + torch.sqrt(Q * A) + 1,
                           v - torch.sqrt(Q * Cc) - 1, v + torch.sqrt(Q * Cc) + 1], 1)
    return terms, box


def _lists64(terms, box, C, ts=16):
    """Per-tile lists in depth order: (item of every pair, start and length per tile)."""
    W, H = C["W"], C["H"]
    tx, ty = (W + ts - 1) // ts, (H + ts - 1) // ts
    ok = (box[:, 0] <= W) & (box[:, 1] >= 0) & (box[:, 2] <= H) & (box[:, 3] >= 0)
    items = ok.nonzero()[:, 0]
    items = items[torch.sort(terms["z"].detach()[items], stable=True)[1]]
    b = box[items]
    x0, x1 = (b[:, 0] / ts).floor().clamp(0, tx - 1).long(), (b[:, 1] / ts).floor().clamp(0, tx - 1).long()
    y0, y1 = (b[:, 2] / ts).floor().clamp(0, ty - 1).long(), (b[:, 3] / ts).floor().clamp(0, ty - 1).long()
    cnt = (x1 - x0 + 1) * (y1 - y0 + 1)
    owner = torch.repeat_interleave(torch.arange(items.numel(), device="cuda"), cnt)
    r = torch.arange(owner.numel(), device="cuda") - (cnt.cumsum(0) - cnt)[owner]
    wid = (x1 - x0 + 1)[owner]
    tile = (y0[owner] + r // wid) * tx + x0[owner] + r % wid
    tile, order = torch.sort(tile, stable=True)
    length = torch.bincount(tile, minlength=tx * ty)
    return items[owner[order]], length.cumsum(0) - length, length, tx, ty


def _sweep64(terms, lists, C, dl, dlsum, out, ts=16, step=32, tiles_at_once=1500):
    """Front-to-back blending of every tile.  With ``dl`` (output gradients
    per pixel and the pixel's total sum of X_i w_i plus its background term)
    the gradients of ``terms`` are added into ``out``; otherwise the blended
    channels and the final transmittance of every pixel are written there."""
    pair, start, length, tx, ty = lists
    t = {k: x.detach() for k, x in terms.items()}
    chan = torch.cat([t["rgb"], t["z"][:, None], torch.ones_like(t["z"])[:, None]]
                     + ([t["feat"]] if "feat" in t else []), 1)
    k = torch.arange(ts * ts, device="cuda")
    for first in range(0, tx * ty, tiles_at_once):
        tid = torch.arange(first, min(first + tiles_at_once, tx * ty), device="cuda")
        px = (tid % tx)[:, None] * ts + k % ts
        py = (tid // tx)[:, None] * ts + k // ts
        inside = (px < C["W"]) & (py < C["H"])
        pix = torch.where(inside, py * C["W"] + px, C["W"] * C["H"])  # one spare pixel takes the outside
        T = torch.ones(px.shape, dtype=F64, device="cuda")
        live = inside.clone()
        acc = torch.zeros(px.shape[0], px.shape[1], chan.shape[1], dtype=F64, device="cuda")
        if dl is not None:
            g, S = dl[pix], dlsum[pix]
        act = torch.arange(tid.numel(), device="cuda")
        for j in range(0, int(length[tid].max()) if tid.numel() else 0, step):
            act = act[(length[tid[act]] > j) & live[act].any(1)]
            if act.numel() == 0:
                break
            at = torch.arange(j, j + step, device="cuda")
            have = at < length[tid[act]][:, None]
            m = pair[torch.where(have, start[tid[act]][:, None] + at, 0)]
            dx = (px[act] + 0.5)[:, None, :] - t["u"][m][:, :, None]
            dy = (py[act] + 0.5)[:, None, :] - t["v"][m][:, :, None]
            a, b, c = (t[q][m][:, :, None] for q in "abc")
            G = torch.exp(-0.5 * (a * dx * dx + c * dy * dy) - b * dx * dy)
            raw = t["o"][m][:, :, None] * G
            hit = (raw >= 1 / 255) & have[:, :, None] & live[act][:, None, :]
            alpha = torch.where(hit, raw.clamp_max(0.99), 0.0)
            after = T[act][:, None, :] * torch.cumprod(1 - alpha, 1)
            hit &= after >= 1e-4
            alpha = torch.where(hit, alpha, 0.0)
            before = after / (1 - alpha)
            w = alpha * before
            if dl is None:
                acc[act] += torch.bmm(w.transpose(1, 2), chan[m])
            else:
                X = torch.bmm(chan[m], g[act].transpose(1, 2))
                xw = torch.cumsum(X * w, 1)
                da = torch.where(hit, before * X - (S[act][:, None, :] - xw) / (1 - alpha), 0.0)
                S[act] -= xw[:, -1]
                da = torch.where(raw <= 0.99, da, 0.0)
                dp = da * raw
                put = lambda name, v: out[name].index_add_(0, m.reshape(-1), v.sum(2).reshape(-1))  # noqa: E731
                put("o", da * G)
                put("u", dp * (a * dx + b * dy))
                put("v", dp * (b * dx + c * dy))
                put("a", -0.5 * dp * dx * dx)
                put("b", -dp * dx * dy)
                put("c", -0.5 * dp * dy * dy)
                out["chan"].index_add_(0, m.reshape(-1), torch.bmm(w, g[act]).reshape(-1, chan.shape[1]))
            stopped = (after < 1e-4).any(1)
            T[act] = T[act] * torch.prod(1 - alpha, 1)
            live[act] &= ~stopped
        if dl is None:
            out["chan"][pix.reshape(-1)] = acc.reshape(-1, chan.shape[1])
            out["T"][pix.reshape(-1)] = T.reshape(-1)


def _sky64(sky, cam, C):
    """Background of every pixel from the cube map."""
    W, H = C["W"], C["H"]
    j = cam["sky_jitter"].to(F64)
    xs = torch.arange(W, device="cuda", dtype=F64)[None, :] + 0.5 + j[0]
    ys = torch.arange(H, device="cuda", dtype=F64)[:, None] + 0.5 + j[1]
    d = torch.stack([(xs - C["cx"]) / C["fx"], (ys - C["cy"]) / C["fy"], torch.ones_like(xs)], -1) @ C["Rm"]
    ax = d.abs()
    main = torch.where((ax[..., 0] >= ax[..., 1]) & (ax[..., 0] >= ax[..., 2]), 0,
                       torch.where(ax[..., 1] >= ax[..., 2], 1, 2))
    x, y, z = d.unbind(-1)
    pos = torch.gather(d, -1, main[..., None])[..., 0] > 0
    face = 2 * main + torch.where(pos, 0, 1)
    sgn = torch.where(pos, 1.0, -1.0).to(F64)
    sc = torch.where(main == 0, -sgn * z, torch.where(main == 1, x, sgn * x))
    tc = torch.where(main == 1, sgn * z, -y)
    ma = torch.gather(ax, -1, main[..., None])[..., 0]
    res = sky.shape[1]
    gx, gy = 0.5 * (sc / ma + 1) * res - 0.5, 0.5 * (tc / ma + 1) * res - 0.5
    x0, y0 = gx.floor(), gy.floor()
    fx, fy = (gx - x0)[..., None], (gy - y0)[..., None]
    at = lambda yy, xx: sky[face, yy.clamp(0, res - 1).long(), xx.clamp(0, res - 1).long()]  # noqa: E731
    return ((1 - fx) * (1 - fy) * at(y0, x0) + fx * (1 - fy) * at(y0, x0 + 1)
            + (1 - fx) * fy * at(y0 + 1, x0) + fx * fy * at(y0 + 1, x0 + 1))


def _render64(P, cam, degree, feats=0, dl_of=None):
    """The images of one view and, with ``dl_of(images)`` giving their output
    gradients, the gradients of P's tensors added into their ``.grad``."""
    C = _cam64(cam)
    W, H = C["W"], C["H"]
    with torch.set_grad_enabled(dl_of is not None):
        terms, box = _project64(P, C, degree, feats)
        f = _sky64(P["sky"], cam, C).reshape(-1, 3) if "sky" in P else None
    with torch.no_grad():
        lists = _lists64(terms, box, C)
        n_chan = 5 + (terms["feat"].shape[1] if feats else 0)
        o = dict(chan=torch.zeros(W * H + 1, n_chan, dtype=F64, device="cuda"),
                 T=torch.ones(W * H + 1, dtype=F64, device="cuda"))
        _sweep64(terms, lists, C, None, None, o)
        chan, T = o["chan"][:-1], o["T"][:-1]
        back = T[:, None] * C["bg"] if f is None else (1 - chan[:, 4:5]) * f
        images = dict(rgb=(chan[:, :3] + back).T.reshape(3, H, W), depth=chan[:, 3].reshape(H, W),
                      alpha=chan[:, 4].reshape(H, W))
        if feats:
            images["feat"] = chan[:, 5:].T.reshape(-1, H, W)
    if dl_of is None:
        return images
    dl = dl_of(images)
    with torch.no_grad():
        flat = lambda k, c: (dl[k].to(F64).reshape(c, -1).T if dl.get(k) is not None  # noqa: E731
                             else torch.zeros(W * H, c, dtype=F64, device="cuda"))
        g = torch.cat([flat("rgb", 3), flat("depth", 1), flat("alpha", 1)]
                      + ([flat("feat", n_chan - 5)] if feats else []), 1)
        if f is not None:
            g[:, 4] -= (g[:, :3] * f).sum(1)
        total = (g * chan).sum(1)
        if f is None:
            total += T * (g[:, :3] * C["bg"]).sum(1)
        pad = lambda x: torch.cat([x, torch.zeros_like(x[:1])])  # noqa: E731
        gt = {k: torch.zeros_like(terms[k]) for k in ("u", "v", "a", "b", "c", "o")}
        gt["chan"] = torch.zeros(terms["u"].numel(), n_chan, dtype=F64, device="cuda")
        _sweep64(terms, lists, C, pad(g), pad(total), gt)
    parts = [(terms[k], gt[k]) for k in ("u", "v", "a", "b", "c", "o")]
    parts += [(terms["rgb"], gt["chan"][:, :3]), (terms["z"], gt["chan"][:, 3])]
    if feats:
        parts.append((terms["feat"], gt["chan"][:, 5:]))
    if f is not None:
        parts.append((f, (1 - chan[:, 4:5]) * g[:, :3]))
    torch.autograd.backward([x for x, _ in parts], [y for _, y in parts])
    return images


def _rgb_loss64(x, y, lam=0.2):
    w = torch.exp(-(torch.arange(11, device="cuda", dtype=F64) - 5) ** 2 / 4.5)
    w = w / w.sum()

    def blur(a):
        h, wd = a.shape[1:]
        a = torch.nn.functional.pad(a, (5, 5, 5, 5))
        a = sum(w[k] * a[:, :, k:k + wd] for k in range(11))
        return sum(w[k] * a[:, k:k + h] for k in range(11))

    mx, my = blur(x), blur(y)
    vx, vy, cxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * cxy + c2) / ((mx * mx + my * my + c1) * (vx + vy + c2))).mean()
    l1 = (x - y).abs().mean()
    return torch.stack([(1 - lam) * l1 + lam * (1 - ssim), l1, ssim])


def _rgb_loss_grad64(x, y):
    x = x.detach().to(F64).requires_grad_(True)
    with torch.enable_grad():
        loss = _rgb_loss64(x, y.to(F64))
        dl, = torch.autograd.grad(loss[0], x)
    return loss.detach(), dl


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort":
        return None  # whole numbers
    d = _inputs(case, seed)
    if kind == "loss":
        loss, dl = _rgb_loss_grad64(d["pred"], d["target"])
        return dict(loss=loss, dl=dl)
    to64 = lambda s: {k: v.to(F64) for k, v in s.items()}  # noqa: E731
    if kind in ("multi", "serve"):
        scenes = [to64(s) for s in d["scenes"]]
        if kind == "serve":
            return [_render64(scenes[k], cam, case["degree"])["rgb"] for k, cam in d["reqs"]]
        return [_render64(scenes[v % 2], cam, case["degree"]) for v, cam in enumerate(d["cams"])]
    P = to64(d["scene"])
    if kind == "forward":
        return [_render64(P, cam, case["degree"]) for cam in d["cams"]]
    for v in P.values():
        v.requires_grad_(True)
    losses = []

    def dl_of(v):
        def f(images):
            if kind == "graph":
                diff = images["rgb"] - d["targets"][v].to(F64)
                losses.append(diff.abs().mean())
                return dict(rgb=diff.sign() / diff.numel())
            if kind == "step":
                loss, dl = _rgb_loss_grad64(images["rgb"], d["targets"][v])
                losses.append(loss)
                return dict(rgb=dl)
            return d["dl"]
        return f

    feats = 1 if kind == "features" else 0
    images = [_render64(P, cam, case["degree"], feats, dl_of(v)) for v, cam in enumerate(d["cams"])]
    grads = {k: v.grad for k, v in P.items()}
    if kind == "autograd":
        return dict(images[0], grads=grads)
    if kind == "graph":
        return dict(images=images, losses=torch.stack(losses), grads=grads)
    if kind == "step":
        return dict(images=images[0], loss=losses[0], grads=grads)
    return dict(images=images[0], grads=grads)

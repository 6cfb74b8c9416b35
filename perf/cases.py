"""Workloads of the UniGS rasterizer, as a program that uses this package runs them.

A case is a dict of plain values; ``kind`` says which public call it makes:

* ``view``: ``Renderer.forward`` - preprocess, binning, composite, normal from
  depth (a viewer, or rendering a trajectory).  ``reuse`` keeps the caller's
  output buffers and skips the instance read-back, as a serving loop does;
  without it the call is the plain ``renderer.forward()``.
* ``step``: ``Renderer.forward`` + ``Renderer.backward`` with upstream
  gradients on every output channel (an optimisation loop with its own loss).
* ``autograd``: ``rasterizer.render`` under torch autograd.
* ``train``: ``Trainer.step`` - render, combined loss, backward, Adam.
* ``loss``: ``Renderer.loss`` on rendered maps.
* ``decode`` / ``decode_bwd``: the anchor MLPs (``DeviceAnchors``) and their
  backward.

The scenes are the package's synthetic rooms and slab (``scenes.py``): the
same distributions, drawn on the GPU so that millions of Gaussians take
milliseconds.  Dense rooms have heavy-tailed sizes (log-normal, sigma 1), as
trained scenes do; the smaller ones are the indoor sizes of the paper's
tables.
"""
from __future__ import annotations

import math

import torch

from paper_2510_12174_gb300 import rasterizer as rz
from paper_2510_12174_gb300 import scenes
from paper_2510_12174_gb300 import train as tr
from paper_2510_12174_gb300.anchors import DeviceAnchors

DEV = "cuda"
Y00 = 0.28209479177387814
PARAMS = ("mean", "quat", "scale", "opacity", "kfac", "sh", "sem")
MAPS = ("rgb", "depth", "normal_g", "kmap", "logits", "normal_d")
MIXED = ((640, 480), (1280, 720), (1920, 1080))


# ------------------------------------------------------------------- the cases
def _case(name, kind, scene, n, w, h, views, sem, deg, bf16, reuse=False, mixed=False):
    return {"name": name, "kind": kind, "scene": scene, "n": n, "width": w, "height": h,
            "views": views, "sem": sem, "sh_degree": deg, "bf16": bf16, "reuse": reuse,
            "mixed": mixed}


def _anchors(name, kind, n, offsets, sem, bf16):
    return {"name": name, "kind": kind, "n": n, "offsets": offsets, "sem": sem, "bf16": bf16}


def listed():
    return [
        # the smallest render: a preview of an object-sized scene, where launches
        # and host work count
        _case("view_256_10k", "view", "slab", 10_000, 256, 256, 1, 16, 0, False),
        # one frame of an interactive viewer on a full room
        _case("view_720p_1M", "view", "dense", 1_000_000, 1280, 720, 1, 64, 3, True, reuse=True),
        # evaluation: a trajectory of cameras of mixed resolution in one batch
        _case("views_mixed_3M", "view", "dense", 3_000_000, 0, 0, 16, 64, 3, True, reuse=True,
              mixed=True),
        # a small scene optimised through autograd at odd image sizes, few classes
        _case("autograd_odd_50k", "autograd", "room", 50_000, 333, 251, 2, 5, 1, False),
        # an indoor scene of the paper's size, one VGA view per iteration, FP32 features
        _case("step_480p_200k", "step", "room", 200_000, 640, 480, 1, 32, 3, False),
        # the headline: batched forward + backward of 16 views, BF16 features
        _case("step_16x720p_1M", "step", "dense", 1_000_000, 1280, 720, 16, 64, 3, True,
              reuse=True),
        # a whole training iteration at the largest size
        _case("train_8x1080p_6M", "train", "dense", 6_000_000, 1920, 1080, 8, 64, 3, True),
        # the combined loss and its gradients on eight full-HD views
        _case("loss_8x1080p", "loss", "room", 1_000, 1920, 1080, 8, 64, 0, True),
        # attribute prediction of an anchor scene: 1M Gaussians for the renderer
        _anchors("decode_100k", "decode", 100_000, 10, 64, True),
        # its backward in training
        _anchors("decode_bwd_100k", "decode_bwd", 100_000, 10, 64, True),
        # a small anchor set, FP32 features, sizes that divide nothing
        _anchors("decode_bwd_3k", "decode_bwd", 3_333, 7, 21, False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "step", "step", "autograd", "loss", "decode",
                       "decode_bwd"])
    if kind in ("decode", "decode_bwd"):
        return {"kind": kind, "n": _log_int(rng, 500, 150_000), "offsets": rng.randint(4, 16),
                "sem": rng.choice([0, rng.randint(1, 64), 64]), "bf16": rng.random() < 0.5}
    w = _log_int(rng, 120, 1920)
    h = max(64, int(w * rng.uniform(0.5, 0.8)))
    if kind == "loss":
        return {"kind": kind, "scene": "room", "n": 500, "width": w, "height": h,
                "views": rng.randint(1, 8), "sem": rng.randint(0, 64), "sh_degree": 0,
                "bf16": False, "reuse": False, "mixed": False}
    n = _log_int(rng, 5_000, 1_500_000)
    bf16 = rng.random() < 0.5
    return {"kind": kind, "scene": "dense" if n > 400_000 else "room", "n": n, "width": w,
            "height": h, "views": rng.randint(1, 4), "sem": rng.choice([0, rng.randint(1, 64), 64]),
            "sh_degree": rng.randint(0, 3), "bf16": bf16, "reuse": rng.random() < 0.5,
            "mixed": False}


# ------------------------------------------------------------------ the inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo


def _randn(g, *shape, mean=0.0, std=1.0):
    return torch.randn(*shape, generator=g, device=DEV) * std + mean


def _room_points(g, n):
    """[3, n] points within 5 cm of the walls of a 6 x 3 x 6 m room and of ten
    boxes on its floor, in proportion to area."""
    hx, hy, hz = (float(x) for x in scenes.ROOM_HALF)
    rects = [((-hx, -hy, -hz), (0, 2 * hy, 0), (0, 0, 2 * hz)),
             ((hx, -hy, -hz), (0, 2 * hy, 0), (0, 0, 2 * hz)),
             ((-hx, -hy, -hz), (2 * hx, 0, 0), (0, 0, 2 * hz)),
             ((-hx, hy, -hz), (2 * hx, 0, 0), (0, 0, 2 * hz)),
             ((-hx, -hy, -hz), (2 * hx, 0, 0), (0, 2 * hy, 0)),
             ((-hx, -hy, hz), (2 * hx, 0, 0), (0, 2 * hy, 0))]
    box = torch.rand(10, 5, generator=g, device=DEV).cpu().tolist()
    for a, b, c, d, e in box:
        sx, sy, sz = 0.2 + 0.8 * a, 0.2 + 0.8 * b, 0.2 + 0.8 * c
        x0, z0 = -hx + d * (2 * hx - sx), -hz + e * (2 * hz - sz)
        y0 = hy - sy
        rects += [((x0, y0, z0), (sx, 0, 0), (0, 0, sz)), ((x0, y0, z0), (0, sy, 0), (0, 0, sz)),
                  ((x0 + sx, y0, z0), (0, sy, 0), (0, 0, sz)),
                  ((x0, y0, z0), (sx, 0, 0), (0, sy, 0)),
                  ((x0, y0, z0 + sz), (sx, 0, 0), (0, sy, 0))]
    O, U, V = (torch.tensor([r[k] for r in rects], device=DEV) for k in range(3))
    N = torch.linalg.cross(U, V)
    area = torch.linalg.vector_norm(N, dim=1)
    which = torch.multinomial(area, n, replacement=True, generator=g)
    P = O[which] + _rand(g, n, 1) * U[which] + _rand(g, n, 1) * V[which] + \
        _rand(g, n, 1, lo=-0.05, hi=0.05) * (N / area[:, None])[which]
    return P.T.contiguous()


def _gaussians(case, g):
    n, c, deg = case["n"], case["sem"], case["sh_degree"]
    feat = torch.bfloat16 if case["bf16"] else torch.float32
    n_sh = (deg + 1) ** 2
    if case["scene"] == "slab":
        mean = torch.stack([_rand(g, n, lo=-1, hi=1), _rand(g, n, lo=-1, hi=1),
                            _rand(g, n, lo=2, hi=6)])
        log_s = _randn(g, 3, n, mean=-4.0, std=0.5)
        sh = torch.zeros(n, n_sh, 3, device=DEV)
        sh[:, 0] = (_rand(g, n, 3) - 0.5) / Y00
    else:
        mean = _room_points(g, n)
        if case["scene"] == "dense":
            log_s = _randn(g, 3, n, mean=-4.5, std=1.0).clamp_(max=-1.0)
        else:
            # the fewer Gaussians cover the same walls, the larger they are
            log_s = _randn(g, 3, n, mean=-2.6 - 0.4 * math.log(max(n, 2000) / 8000.0), std=0.5)
        sh = _randn(g, n, n_sh, 3, std=0.2)
    quat = _randn(g, 4, n)
    quat = quat / torch.linalg.vector_norm(quat, dim=0) * _rand(g, 1, n, lo=0.5, hi=2.0)
    return {"mean": mean, "quat": quat.contiguous(), "scale": torch.exp(log_s),
            "opacity": torch.sigmoid(_randn(g, n)), "kfac": torch.sigmoid(_randn(g, n, mean=2.0)),
            "sh": sh.to(feat).contiguous(), "sem": _randn(g, n, c).to(feat)}


def _cameras(case, seed):
    if case["scene"] == "slab":
        return [scenes.front_camera(case["width"], case["height"], float(case["width"]))]
    if case["mixed"]:
        res = MIXED
    else:
        res = [(case["width"], case["height"])]
    return scenes.orbit_cameras(case["views"], seed=int(seed) % 1000, resolutions=res)


def _pixels(case):
    if not case["mixed"]:
        return case["width"] * case["height"] * case["views"]
    return sum(c.width * c.height for c in _cameras(case, 0))


def _channels(n_sem):
    return {"rgb": 3, "depth": 1, "normal_g": 3, "kmap": 1, "logits": n_sem, "normal_d": 3}


def _upstream(g, P, n_sem):
    """Upstream gradients of every map.  A loss gives the two normal maps a small
    weight: one is a difference of depths, the other has the unbounded
    derivative of an ellipsoid's outline."""
    return {k: _randn(g, c * P, std=0.01 if k.startswith("normal") else 1.0)
            for k, c in _channels(n_sem).items()}


def _targets(g, P, n_sem):
    """Per-pixel training targets: colours, depths with unmeasured pixels (0),
    normals (unit length on average), labels with unlabelled pixels (-1)."""
    depth = _rand(g, P, lo=1.0, hi=4.0)
    depth[_rand(g, P) < 0.15] = 0.0
    label = torch.randint(0, max(n_sem, 1), (P,), generator=g, device=DEV, dtype=torch.int32)
    label[_rand(g, P) < 0.1] = -1
    normal = _randn(g, 3 * P)
    return {"rgb": _rand(g, 3 * P), "depth": depth, "normal": normal / math.sqrt(3.0),
            "label": label}


def _anchor_inputs(case, g):
    n, m, c = case["n"], case["offsets"], case["sem"]
    pos = torch.stack([_rand(g, n, lo=-1.5, hi=1.5), _rand(g, n, lo=-1, hi=1),
                       _rand(g, n, lo=2, hi=5)])
    outs = {"sem": c, "k": 1, "opacity": m, "color": 3 * m, "cov": 7 * m}
    mlps = {k: {"w1": _randn(g, 32, 32, std=1 / math.sqrt(32.0)), "b1": _randn(g, 32, std=0.1),
                "w2": _randn(g, o, 32, std=0.25), "b2": _randn(g, o, std=0.1)}
            for k, o in outs.items() if o}
    arrays = {"pos": pos, "scale": torch.exp(_randn(g, 3, n, mean=-2.6, std=0.3)),
              "offsets": _randn(g, n, m, 3), "feat": _randn(g, n, 32), "sem": _randn(g, n, c),
              "kfac": _rand(g, n, lo=0.8, hi=1.2)}
    N = n * m
    up = {"mean": _randn(g, 3, N), "quat": _randn(g, 4, N), "scale": _randn(g, 3, N),
          "opacity": _randn(g, N), "kfac": _randn(g, N), "sh": _randn(g, N, 1, 3),
          "sem": _randn(g, N, c)}
    return arrays, mlps, up


def _loss_maps(g, P, n_sem):
    normal = _randn(g, 3 * P) / math.sqrt(3.0)
    normal[_rand(g, 3 * P) < 0.1] = 0.0
    return {"rgb": _rand(g, 3 * P), "depth": _rand(g, P, lo=1, hi=4), "normal_d": normal,
            "normal_g": torch.zeros(3 * P, device=DEV), "kmap": _rand(g, P, lo=0.5, hi=1.5),
            "logits": _randn(g, n_sem * P, std=2.0), "T_final": torch.zeros(P, device=DEV),
            "n_contrib": torch.zeros(P, dtype=torch.int32, device=DEV)}


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("decode", "decode_bwd"):
        arrays, mlps, up = _anchor_inputs(case, g)
        anchors = DeviceAnchors(arrays["pos"], arrays["scale"], arrays["offsets"], arrays["feat"],
                                arrays["sem"], arrays["kfac"], mlps)
        st = {"kind": kind, "anchors": anchors, "bf16": case["bf16"]}
        if kind == "decode":
            st["out"] = anchors.decode(case["bf16"])
        else:
            st["up"], st["grads"] = up, anchors.alloc_grads()
        return st
    G = _gaussians(case, g)
    cams = _cameras(case, seed)
    P = sum(c.width * c.height for c in cams)
    if kind == "train":
        raw = {"mean": G["mean"], "quat": G["quat"], "log_scale": torch.log(G["scale"]),
               "logit_opacity": torch.logit(G["opacity"], 1e-6), "k": G["kfac"],
               "sh": G["sh"].float(), "sem": G["sem"].float()}
        trainer = tr.Trainer(raw, case["sh_degree"], cams, _targets(g, P, case["sem"]),
                             tr.TrainConfig(feat_bf16=case["bf16"]))
        return {"kind": kind, "trainer": trainer}
    scene = rz.DeviceScene(*(G[k] for k in PARAMS), case["sh_degree"])
    r = rz.Renderer(scene, cams)
    st = {"kind": kind, "renderer": r, "reuse": case["reuse"]}
    if case["reuse"]:
        # the first frame sizes the renderer's plan; later ones never read back
        st["out"] = r.forward()
    if kind == "loss":
        st["maps"] = _loss_maps(g, P, case["sem"])
        st["targets"] = _targets(g, P, case["sem"])
        st["record"] = torch.zeros(16, device=DEV)
        st["lgrads"] = r.alloc_loss_grads()
    if kind in ("step", "autograd"):
        st["up"] = _upstream(g, P, case["sem"])
        if case["reuse"]:
            st["grads"] = r.alloc_grads()
            st["g_depth"] = torch.empty(P, device=DEV)
    if kind == "autograd":
        for k in PARAMS:
            getattr(scene, k).requires_grad_(True)
    return st


# ------------------------------------------------------------------- the calls
def run(state):
    kind = state["kind"]
    if kind == "decode":
        d = state["anchors"].decode(state["bf16"], out=state["out"])
        return {k: getattr(d, k) for k in PARAMS}
    if kind == "decode_bwd":
        return state["anchors"].decode_backward(state["up"], state["grads"])
    if kind == "train":
        t = state["trainer"]
        t.step()
        return {"record": t.record, "out": t.out, "grads": t.grads}
    r = state["renderer"]
    if kind == "loss":
        r.loss(state["maps"], state["targets"], state["record"], state["lgrads"])
        return {"record": state["record"], "grads": state["lgrads"]}
    if kind == "autograd":
        s = r.scene
        out = rz.render(r)
        up = state["up"]
        leaves = [getattr(s, k) for k in PARAMS]
        grads = torch.autograd.grad(out, leaves, [up[k] for k in MAPS])
        return {"out": dict(zip(MAPS, out)), "grads": dict(zip(PARAMS, grads))}
    if state["reuse"]:
        out = r.forward(state["out"], readback=False)
    else:
        out = r.forward()
    if kind == "view":
        return out
    grads = r.backward(out, state["up"], grads=state.get("grads"), g_depth_buf=state.get("g_depth"))
    return {"out": out, "grads": grads}


# -------------------------------------------------------------------- the work
def _blended_per_pixel(case):
    """Gaussians blended per pixel: measured on the room scenes (about 150 where
    the walls are opaque), fewer where the Gaussians do not cover the image."""
    if case["scene"] == "slab":
        return 20
    return 150 if case["scene"] == "dense" else 40


def work(case):
    kind, n, c = case["kind"], case["n"], case["sem"]
    e = 2 if case["bf16"] else 4
    if kind in ("decode", "decode_bwd"):
        m = case["offsets"]
        anchor = 4 * (3 + 3 + 3 * m + 32 + c + 1)
        gauss = 4 * 12 + (4 * (3 + c) if kind == "decode_bwd" else e * (3 + c))
        outs = c + 1 + m + 3 * m + 7 * m
        macs = 32 * 32 * (5 if c else 4) + 32 * outs
        if kind == "decode":
            return {"bytes": n * (anchor + m * gauss), "flops": 2 * n * macs}
        return {"bytes": n * (2 * anchor + m * gauss), "flops": 6 * n * macs}
    P = _pixels(case)
    if kind == "loss":
        return {"bytes": P * 4 * (2 * (8 + c) + 8), "flops": P * (30 + 8 * c)}
    params = n * (48 + e * (3 * (case["sh_degree"] + 1) ** 2 + c))
    grads = n * 4 * (12 + 3 * (case["sh_degree"] + 1) ** 2 + c)
    maps = P * 4 * (13 + c)
    pairs = P * _blended_per_pixel(case)
    fwd = pairs * (114 + 2 * (11 + c))
    if kind == "view":
        return {"bytes": params + maps, "flops": fwd}
    w = {"bytes": params + 2 * maps + grads, "flops": fwd + pairs * (310 + 4 * c)}
    if kind == "train":
        w["bytes"] += P * 32 + 5 * grads  # targets; Adam reads raw, m, v and writes them
    return w


# --------------------------------------------------- the same in 64 bits, plainly
D = torch.float64


def _basis(d, deg):
    x, y, z = d.unbind(-1)
    pi = math.pi
    b = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg >= 1:
        k = math.sqrt(3 / (4 * pi))
        b += [k * y, k * z, k * x]
    if deg >= 2:
        k = 0.5 * math.sqrt(15 / pi)
        b += [k * x * y, k * y * z, 0.25 * math.sqrt(5 / pi) * (3 * z * z - 1), k * x * z,
              0.5 * k * (x * x - y * y)]
    if deg >= 3:
        k1, k2 = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi)
        k3, k4 = 0.25 * math.sqrt(21 / (2 * pi)), 0.25 * math.sqrt(7 / pi)
        b += [k1 * y * (3 * x * x - y * y), k2 * x * y * z, k3 * y * (5 * z * z - 1),
              k4 * z * (5 * z * z - 3), k3 * x * (5 * z * z - 1), 0.5 * k2 * z * (x * x - y * y),
              k1 * x * (x * x - 3 * y * y)]
    return torch.stack(b, -1)


def _t64(x):
    return torch.as_tensor(x, dtype=D, device=DEV)


# columns of the per-Gaussian matrix that the composite reads
_COLS = {"m": (0, 2), "con": (2, 5), "op": (5, 6), "rgb": (6, 9), "R": (9, 18), "s": (18, 21),
         "vs": (21, 24), "k": (24, 25), "sem": (25, None)}


def _project(G, deg, cam):
    """Per-Gaussian quantities of one camera: the matrix of _COLS, and (without
    derivative) 3-sigma radius, depth and visibility."""
    R_wc, t, C = _t64(cam.R_wc), _t64(cam.t_wc), _t64(cam.C)
    mu = G["mean"].T
    x, y, z = (mu @ R_wc.T + t).unbind(-1)
    q = G["quat"] / torch.linalg.vector_norm(G["quat"], dim=0)
    qw, qx, qy, qz = q
    R = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                     2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                     2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)],
                    -1).reshape(-1, 3, 3)
    s = G["scale"].T
    front = (z > cam.z_near).detach()
    zs = torch.where(front, z, torch.ones_like(z))
    zero = torch.zeros_like(z)
    J = torch.stack([cam.fx / zs, zero, -cam.fx * x / zs ** 2, zero, cam.fy / zs,
                     -cam.fy * y / zs ** 2], -1).reshape(-1, 2, 3)
    V = J @ R_wc @ (R * s[:, None, :])
    cov = V @ V.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * c - b * b
    dirs = mu - C
    dirs = dirs / torch.linalg.vector_norm(dirs, dim=1, keepdim=True)
    rgb = (torch.einsum("nk,nkc->nc", _basis(dirs, deg), G["sh"]) + 0.5).clamp(min=0)
    vs = torch.einsum("nji,nj->ni", R, C - mu) / s
    M = torch.cat([torch.stack([cam.fx * x / zs + cam.cx, cam.fy * y / zs + cam.cy, c / det,
                                -b / det, a / det, G["opacity"]], -1), rgb, R.reshape(-1, 9), s, vs,
                   G["kfac"][:, None], G["sem"]], 1)
    with torch.no_grad():
        mid = 0.5 * (a + c)
        lam = mid + torch.sqrt((mid * mid - det).clamp(min=0.1))
        rad = torch.ceil(3 * torch.sqrt(lam))
    return M, rad, z.detach(), front & (det > 0).detach()


def _composite(A, rad, uv, cam):
    """Front-to-back blend of the ordered Gaussians A [L, F] at the pixels uv."""
    f = {k: A[:, i:j] for k, (i, j) in _COLS.items()}
    d = uv[:, None, :] - f["m"][None]
    dx, dy = d[..., 0], d[..., 1]
    con = f["con"]
    alpha = (f["op"][:, 0] * torch.exp(-0.5 * (con[:, 0] * dx * dx + con[:, 2] * dy * dy) -
                                       con[:, 1] * dx * dy)).clamp(max=0.99)
    with torch.no_grad():
        drawn = (alpha >= 1 / 255) & (d.abs().amax(-1) <= rad)
        drawn &= torch.cumprod(torch.where(drawn, 1 - alpha, torch.ones_like(alpha)), 1) >= 1e-4
    om = torch.where(drawn, 1 - alpha, torch.ones_like(alpha))
    T = torch.cumprod(om, 1)
    w = torch.where(drawn, alpha, torch.zeros_like(alpha)) * \
        torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    ray = torch.stack([(uv[:, 0] - cam.cx) / cam.fx, (uv[:, 1] - cam.cy) / cam.fy,
                       torch.ones_like(uv[:, 0])], -1) @ _t64(cam.R_cw).T
    R = f["R"].reshape(-1, 3, 3)
    ds = torch.einsum("pj,ljk->plk", ray, R) / f["s"]
    vs = f["vs"][None].expand_as(ds)
    qa, qb = (ds * ds).sum(-1), (vs * ds).sum(-1)
    cv = torch.linalg.cross(vs, ds)
    disc = qa - (cv * cv).sum(-1)
    hit = (disc > 0).detach()
    inside = ((f["vs"] ** 2).sum(-1) <= 1).detach()
    root = torch.where(hit, torch.where(hit, disc, torch.ones_like(disc)).sqrt(),
                       torch.zeros_like(disc))
    p = vs + ((torch.where(inside, root, -root) - qb) / qa)[..., None] * ds
    nrm = torch.einsum("lij,plj->pli", R, p / f["s"])
    nrm = nrm / torch.linalg.vector_norm(nrm, dim=-1, keepdim=True)
    nrm = torch.where(inside[None, :, None], -nrm, nrm)
    return {"rgb": w @ f["rgb"], "depth": (w * (-qb / qa)).sum(1)[:, None],
            "normal_g": torch.einsum("pl,plc->pc", w, nrm), "kmap": w @ f["k"],
            "logits": w @ f["sem"], "T_final": T[:, -1:]}


def _depth_normal(depth, cam):
    """Normal map [3, H, W] of a depth map: central differences at 1 and 2
    pixels, fused, normalised, facing the camera."""
    H, W = depth.shape
    v, u = torch.meshgrid(torch.arange(H, dtype=D, device=DEV), torch.arange(W, dtype=D, device=DEV),
                          indexing="ij")
    Pc = torch.stack([(u - cam.cx) / cam.fx * depth, (v - cam.cy) / cam.fy * depth, depth])
    Pw = torch.einsum("ij,jhw->ihw", _t64(cam.R_cw), Pc)

    def at(g):
        if H <= 2 * g or W <= 2 * g:
            return torch.zeros_like(Pw)
        n = torch.linalg.cross(Pw[:, g:H - g, 2 * g:] - Pw[:, g:H - g, :W - 2 * g],
                               Pw[:, 2 * g:, g:W - g] - Pw[:, :H - 2 * g, g:W - g], dim=0)
        return torch.nn.functional.pad(n, (g, g, g, g))

    n1, n2 = at(1), at(2)
    nf = 0.5 * n1 + 0.5 * n2 * torch.where((n1 * n2).sum(0) >= 0, 1.0, -1.0)
    inner = torch.zeros(H, W, dtype=torch.bool, device=DEV)
    inner[2:H - 2, 2:W - 2] = True
    ok = inner & (nf.detach().abs().sum(0) > 0)
    nf = torch.where(ok, nf, torch.ones_like(nf))
    n = torch.where(ok, nf / torch.linalg.vector_norm(nf, dim=0), torch.zeros_like(nf))
    return torch.where((n * -Pw).sum(0) < 0, -n, n)


def _tiles(M, rad, z, vis, cam):
    """(pixel indices, pixel coordinates, ordered Gaussian ids) of each 16 x 16 tile."""
    ids = vis.nonzero()[:, 0]
    ids = ids[torch.sort(z[ids].float(), stable=True).indices]
    m, r = M[ids, :2].detach(), rad[ids]
    lo, hi = m - r[:, None], m + r[:, None]
    seen = (hi >= 0).all(1) & (lo[:, 0] <= cam.width) & (lo[:, 1] <= cam.height)
    ids, lo, hi = ids[seen], lo[seen], hi[seen]
    for y0 in range(0, cam.height, 16):
        y1 = min(y0 + 16, cam.height)
        row = (hi[:, 1] >= y0) & (lo[:, 1] <= y1 - 1)
        rid, rlo, rhi = ids[row], lo[row, 0], hi[row, 0]
        for x0 in range(0, cam.width, 16):
            x1 = min(x0 + 16, cam.width)
            v, u = torch.meshgrid(torch.arange(y0, y1, device=DEV), torch.arange(x0, x1, device=DEV),
                                  indexing="ij")
            sel = rid[(rhi >= x0) & (rlo <= x1 - 1)]
            yield ((v * cam.width + u).reshape(-1),
                   torch.stack([u.reshape(-1), v.reshape(-1)], -1).to(D), sel)


def _exact_render(case, seed, up):
    """The maps, and with upstream gradients `up` the parameter gradients."""
    g = _gen(seed)
    G = {k: v.to(D) for k, v in _gaussians(case, g).items()}
    cams = _cameras(case, seed)
    P = sum(c.width * c.height for c in cams)
    if up:
        up = {k: v.to(D) for k, v in _upstream(g, P, case["sem"]).items()}
        for v in G.values():
            v.requires_grad_(True)
    ch = dict(_channels(case["sem"]), T_final=1)
    maps, off = {k: [] for k in ch}, 0
    for cam in cams:
        H, W = cam.height, cam.width
        M, rad, z, vis = _project(G, case["sh_degree"], cam)
        tiles = list(_tiles(M, rad, z, vis, cam))
        img = {k: torch.zeros(H * W, c, dtype=D, device=DEV) for k, c in ch.items()}
        img["T_final"] += 1
        with torch.no_grad():
            for pix, uv, ids in tiles:
                if len(ids):
                    for k, v in _composite(M[ids], rad[ids], uv, cam).items():
                        img[k][pix] = v
        depth = img["depth"].reshape(H, W).requires_grad_(bool(up))
        img["normal_d"] = _depth_normal(depth, cam).reshape(3, -1).T
        if up:
            cut = {k: up[k][c * off:c * (off + H * W)].reshape(c, H * W).T for k, c in ch.items()
                   if k in up}
            g_depth = cut["depth"] + torch.autograd.grad(
                (img["normal_d"] * cut["normal_d"]).sum(), depth)[0].reshape(-1, 1)
            gM = torch.zeros_like(M)
            for pix, uv, ids in tiles:
                if len(ids):
                    A = M[ids].detach().requires_grad_(True)
                    o = _composite(A, rad[ids], uv, cam)
                    loss = (o["depth"] * g_depth[pix]).sum()
                    for k in ("rgb", "normal_g", "kmap", "logits"):
                        loss = loss + (o[k] * cut[k][pix]).sum()
                    gM.index_add_(0, ids, torch.autograd.grad(loss, A)[0])
            M.backward(gM)
        for k in ch:
            maps[k].append(img[k].detach().T.reshape(-1))
        off += H * W
    maps = {k: torch.cat(v) for k, v in maps.items()}
    maps["n_contrib"] = None
    return maps, {k: v.grad for k, v in G.items()} if up else None


def _exact_loss(case, seed):
    g = _gen(seed)
    _gaussians(case, g)
    views, HW, c = case["views"], case["width"] * case["height"], case["sem"]
    P = views * HW
    o, t = _loss_maps(g, P, c), _targets(g, P, c)
    cut = lambda x, ch, k: x[ch * k * HW:ch * (k + 1) * HW].to(D)
    nd, nl = int((t["depth"] > 0).sum()), int(((t["label"] >= 0) & (t["label"] < c)).sum())
    tot = dict.fromkeys(("l1", "n", "d", "s", "k"), 0.0)
    grad = {k: [] for k in ("rgb", "depth", "normal_d", "kmap", "logits")}
    for k in range(views):
        d = cut(o["rgb"], 3, k) - cut(t["rgb"], 3, k)
        tot["l1"] += float(d.abs().sum()) / (3 * P)
        grad["rgb"].append(d.sign() / (3 * P))
        n = cut(t["normal"], 3, k)
        tot["n"] += float((cut(o["normal_d"], 3, k) * n).sum()) / P
        grad["normal_d"].append(-n / P)
        dt = cut(t["depth"], 1, k)
        d = torch.where(dt > 0, cut(o["depth"], 1, k) - dt, torch.zeros_like(dt))
        tot["d"] += float(d.abs().sum()) / max(nd, 1)
        grad["depth"].append(d.sign() / max(nd, 1))
        d = cut(o["kmap"], 1, k) - 1
        tot["k"] += float(d.abs().sum()) / P
        grad["kmap"].append(d.sign() / P)
        if c:
            lab = t["label"][k * HW:(k + 1) * HW].long()
            has = (lab >= 0).to(D)
            lp = torch.log_softmax(cut(o["logits"], c, k).reshape(c, HW), 0)
            lab = lab.clamp(min=0)[None]
            tot["s"] -= float((lp.gather(0, lab)[0] * has).sum()) / max(nl, 1)
            gr = lp.exp_()
            gr.scatter_add_(0, lab, -torch.ones_like(gr[:1]))
            grad["logits"].append((gr * has / max(nl, 1)).reshape(-1).float())
    L = {"l1": tot["l1"], "n": 1 - tot["n"], "d": tot["d"], "s": tot["s"], "k": tot["k"]}
    w = {k: 0.1 * abs(L["l1"]) / abs(v) if v else 0.0 for k, v in L.items()}
    w["l1"] = 1.0
    rec = [sum(w[k] * L[k] for k in L)] + [L[k] for k in ("l1", "n", "d", "s", "k")] + \
        [w[k] for k in ("l1", "n", "d", "s", "k")] + [nd, nl if c else 0, 0, 0, 0]
    out = {m: torch.cat(grad[m]) * w[k] if grad[m] else torch.zeros(0, device=DEV) for m, k in
           (("rgb", "l1"), ("depth", "d"), ("normal_d", "n"), ("kmap", "k"), ("logits", "s"))}
    return {"record": torch.tensor(rec, dtype=D), "grads": out}


def _exact_decode(case, seed):
    arrays, mlps, up = _anchor_inputs(case, _gen(seed))
    a = {k: v.to(D).requires_grad_(True) for k, v in arrays.items()}
    W = {n: {k: v.to(D).requires_grad_(True) for k, v in m.items()} for n, m in mlps.items()}
    n, m, c = case["n"], case["offsets"], case["sem"]
    N = n * m
    y = {k: torch.relu(a["feat"] @ p["w1"].T + p["b1"]) @ p["w2"].T + p["b2"] for k, p in W.items()}
    sig = torch.sigmoid
    cov = y["cov"].reshape(n, m, 7)
    l = a["scale"].T[:, None, :]
    sem = a["sem"] * sig(y["sem"]) if c else a["sem"]
    out = {"mean": (a["pos"].T[:, None, :] + l * a["offsets"]).reshape(N, 3).T,
           "quat": cov[..., 3:].reshape(N, 4).T, "scale": (l * sig(cov[..., :3])).reshape(N, 3).T,
           "opacity": sig(y["opacity"]).reshape(N),
           "kfac": (a["kfac"][:, None] * sig(y["k"])).expand(n, m).reshape(N),
           "sh": ((sig(y["color"]) - 0.5) / Y00).reshape(N, 1, 3),
           "sem": sem[:, None, :].expand(n, m, c).reshape(N, c)}
    if case["kind"] == "decode":
        return {k: v.detach() for k, v in out.items()}
    sum((v * up[k].to(D)).sum() for k, v in out.items()).backward()
    g = {k: v.grad if v.grad is not None else torch.zeros_like(v) for k, v in a.items()}
    g["mlps"] = {k: {e: v.grad for e, v in p.items()} for k, p in W.items()}
    return g


def exact(case, seed):
    kind = case["kind"]
    if kind in ("decode", "decode_bwd"):
        return _exact_decode(case, seed)
    if kind == "train":
        return None  # minutes in 64 bits
    if kind == "loss":
        return _exact_loss(case, seed)
    tiles = _pixels(case) / 256
    if kind == "view":
        # the whole image tile by tile; a trajectory would take minutes
        return _exact_render(case, seed, None)[0] if tiles <= 8000 else None
    if tiles > 3000:
        return None
    maps, grads = _exact_render(case, seed, True)
    if kind == "autograd":
        maps = {k: maps[k] for k in MAPS}
    return {"out": maps, "grads": grads}

"""The workloads this framework's speed is judged on, through its public Python entry points.

``listed()`` names them and ``draw()`` gives more of the same ranges.  ``prepare`` makes what a user's
program holds before the call (scene, cameras, rasterizer, optimiser, targets) on the GPU from a seed,
``run`` is one pass, ``work`` the bytes and operations a pass cannot do without, and ``exact`` the pass's
outputs in float64 from plain torch, written here from the paper's equations.

Scenes follow the distributions of ``scenes.make_scene`` (clustered Gaussian mixture in [-5, 5]^3 or a
uniform cube, log-uniform scales, logistic-normal opacity) and cameras look at the origin from a sphere;
both are drawn on the device here, so that a new state takes milliseconds.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2510_03312_gb300 import raster
from paper_2510_03312_gb300 import scenes as S
from paper_2510_03312_gb300 import train as TR

DEV = "cuda"
ACT_SIGMOID, ACT_EXP = 1, 2
SIZES = ((256, 192), (400, 301), (640, 360), (800, 600), (1280, 720), (1352, 1014), (1600, 1060), (1920, 1080))


def _view_case(name, kind, N, P, views, width, height, rot=0, layout="clusters", tile_w=16, tile_h=16, form="grid"):
    return {"name": name, "kind": kind, "N": N, "P": P, "views": views, "width": width, "height": height, "rot": rot,
            "layout": layout, "tile_w": tile_w, "tile_h": tile_h, "form": form}


def listed():
    return [
        # interactive preview of a small static asset: latency of one forward render (the static small workload)
        _view_case("preview_4k", "render", 3, 4096, 1, 128, 128, layout="uniform"),
        # playback of a dynamic scene: one frame (camera, time) at full HD, forward only
        _view_case("frame_n7", "render", 7, 300_000, 1, 1920, 1080, rot=1),
        # the flagship: forward and backward of one dense 1600x1060 view of a million static primitives
        _view_case("step_1m", "step", 3, 1_000_000, 1, 1600, 1060),
        # a batch of cameras of a view-dependent scene in one problem, forward and backward
        _view_case("batch_n6", "step", 6, 500_000, 16, 1280, 720),
        # a batch of (camera, time) queries of a dynamic scene, replayed as a captured CUDA graph
        _view_case("graph_n7", "graph", 7, 300_000, 8, 1352, 1014),
        # a capture with very deep tiles (a dense far cluster on one tile), long lists split across CTAs
        _view_case("deep_split", "step", 3, 360_000, 1, 1600, 1060, layout="deep", form="split"),
        # differentiable rendering inside a PyTorch program: the autograd function, ragged views, small scene
        _view_case("autograd_8k", "autograd", 6, 8191, 2, 157, 117, rot=1),
        # a service's uneven queue: many scenes, sizes and resolutions in one batched step
        {"name": "uneven_batch", "kind": "batch", "scenes": 6, "jobs": 32, "p_lo": 10_000, "p_hi": 2_000_000,
         "size_seed": 4, "tile_w": 16, "tile_h": 16},
        # the image loss (L1 + D-SSIM with its gradient) of one training view
        {"name": "loss_1view", "kind": "loss", "views": 1, "width": 1600, "height": 1060},
        # the fused optimiser step of a view-dependent scene with spatial noise, odd primitive count
        {"name": "adam_n6", "kind": "adam", "N": 6, "rot": 1, "P": 500_003, "noise": True},
        # MCMC relocation of the dead primitives of a scene in training
        {"name": "relocate_1m", "kind": "relocate", "N": 3, "rot": 0, "P": 1_000_000, "dead": 0.05},
        # one whole training iteration as trainers run it: a single view, loss, backward, Adam
        _view_case("train_n6", "train", 6, 200_000, 1, 800, 600, layout="clusters"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("render", "step", "step", "graph", "autograd", "batch", "loss", "adam", "relocate", "train"))
    if kind in ("render", "step", "graph", "train"):
        N = rng.choice((3, 4, 6, 7))
        views = 1 if kind == "train" else _log_int(rng, 1, 16)
        w, h = rng.choice(SIZES)
        w, h = w - rng.randrange(16), h - rng.randrange(16)
        P = _log_int(rng, 4000, 1_000_000)
        while P * views > 8_000_000 or w * h * views > 16_000_000:  # at most the largest listed case's records and pixels
            views = max(1, views // 2)
            P = min(P, 8_000_000 // views)
        tw, th = rng.choice(((16, 16), (16, 16), (8, 8), (16, 32), (32, 32)))
        form = rng.choice(("grid", "grid", "grid", "persistent", "split"))
        deep = kind == "step" and views == 1 and N == 3 and P >= 50_000 and rng.random() < 0.3
        layout = "deep" if deep else ("uniform" if P < 20_000 else "clusters")
        return {k: v for k, v in _view_case("", kind, N, P, views, w, h, rot=rng.choice((0, 1)), layout=layout, tile_w=tw,
                                            tile_h=th, form=form).items() if k != "name"}
    if kind == "autograd":
        return {k: v for k, v in _view_case("", kind, rng.choice((3, 4, 6, 7)), _log_int(rng, 500, 50_000), rng.randint(1, 4),
                                            rng.randint(33, 320), rng.randint(33, 240), rot=rng.choice((0, 1))).items()
                if k != "name"}
    if kind == "batch":
        return {"kind": kind, "scenes": rng.randint(2, 6), "jobs": rng.randint(6, 32), "p_lo": 5_000,
                "p_hi": _log_int(rng, 100_000, 1_000_000), "size_seed": rng.randrange(1000), "tile_w": 16, "tile_h": 16}
    if kind == "loss":
        w, h = rng.choice(SIZES)
        return {"kind": kind, "views": rng.randint(1, 4), "width": w - rng.randrange(31), "height": h - rng.randrange(31)}
    N = rng.choice((3, 4, 6, 7))
    if kind == "adam":
        return {"kind": kind, "N": N, "rot": rng.choice((0, 1)), "P": _log_int(rng, 5_000, 1_000_000), "noise": rng.random() < 0.5}
    return {"kind": kind, "N": N, "rot": rng.choice((0, 1)), "P": _log_int(rng, 5_000, 1_000_000),
            "dead": rng.choice((0.01, 0.05, 0.2))}


# ---------------------------------------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _uni(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo


def _log_uni(g, lo, hi, *shape):
    return torch.exp(_uni(g, math.log(lo), math.log(hi), *shape))


def _nrm(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _scene(g, N, P, rot, layout, cam=None):
    """Activated parameters [K, P] in plane order."""
    C = N - 3
    if layout == "uniform":
        mx = _uni(g, -1.0, 1.0, 3, P)
    elif layout == "deep":
        mx = _uni(g, -5.0, 5.0, 3, P)
    else:
        centres = _uni(g, -5.0, 5.0, 3, 64)
        mx = centres[:, torch.randint(0, 64, (P,), generator=g, device=DEV)] + 0.3 * _nrm(g, 3, P)
    sx = _log_uni(g, 0.01, 0.1, 3, P)
    op = torch.sigmoid(_nrm(g, 1, P))
    if layout == "deep":  # a sixth of the primitives small and faint around one point in front of the camera
        R, t = cam
        n = P // 6
        point = (-R.T @ t + 4.0 * R[2]).to(torch.float32).to(DEV)
        mx[:, P - n:] = point[:, None] + 0.01 * _uni(g, -1.0, 1.0, 3, n)
        sx[:, P - n:] = _log_uni(g, 0.002, 0.005, 3, n)
        op[:, P - n:] = torch.sigmoid(-3.0 + 0.3 * _nrm(g, 1, n))
    if rot == 0:
        q = _nrm(g, 4, P)
        r = q / q.norm(dim=0, keepdim=True)
    else:
        r = 0.3 * _nrm(g, 3, P)
    b = 0.5 * _nrm(g, 1 + C, P)
    rgb = _uni(g, 0.0, 1.0, 3, P)
    mq, sq = [], []
    if C in (1, 4):
        mq.append(_uni(g, 0.0, 1.0, 1, P))
        sq.append(_log_uni(g, 0.02, 0.5, 1, P))
    if C >= 3:
        d = _nrm(g, 3, P)
        mq.append(d / d.norm(dim=0, keepdim=True))
        sq.append(_log_uni(g, 0.2, 2.0, 3, P))
    planes = [mx]
    if C:
        sq = torch.cat(sq)
        lqx = (sq[:, None, :] * _uni(g, -0.5, 0.5, C, 3, P)).reshape(3 * C, P)
        lq = torch.cat([(sq[i] if i == j else sq[i] * _uni(g, -0.25, 0.25, P))[None] for i in range(C) for j in range(i + 1)])
        planes += mq + [r, sx, lqx, lq, b, op, rgb]
    else:
        planes += [r, sx, b, op, rgb]
    return torch.cat(planes).contiguous()


def _pose(rng):
    """World-to-camera rotation and translation (float64) of a camera on the radius-8 sphere, y > 0, looking at the origin."""
    u = torch.tensor([rng.gauss(0.0, 1.0) for _ in range(3)], dtype=torch.float64)
    u = u / u.norm()
    u[1] = u[1].abs()
    p = 8.0 * u
    z = -p / p.norm()
    x = torch.linalg.cross(torch.tensor([0.0, 1.0, 0.0], dtype=torch.float64), z)
    x = x / x.norm()
    R = torch.stack([x, torch.linalg.cross(z, x), z])
    return R, -R @ p


def _view(R, t, w, h, time, scene):
    return S.make_view(R.numpy(), t.numpy(), w, h, time=time, scene_id=scene)


def _raster_inputs(case, seed):
    """(scene parameter tensors with their N, views, config) of a render, step, graph, autograd or train case."""
    rng = random.Random(seed)
    g = _gen(seed)
    if case["layout"] == "uniform":  # the cube of half-width 1 seen from distance 3
        poses = [(torch.eye(3, dtype=torch.float64), torch.tensor([0.0, 0.0, 3.0], dtype=torch.float64) + 0.1 * i)
                 for i in range(case["views"])]
    else:
        poses = [_pose(rng) for _ in range(case["views"])]
    views = [_view(R, t, case["width"], case["height"], rng.random(), 0) for R, t in poses]
    params = _scene(g, case["N"], case["P"], case["rot"], case["layout"], poses[0])
    cfg = S.RasterConfig(tile_w=case["tile_w"], tile_h=case["tile_h"], persistent=case["form"] == "persistent",
                         split_lists=case["form"] == "split")
    return [(case["N"], case["rot"], params)], views, cfg


def _batch_sizes(case):
    """Scene (N, rotation, P) and job (width, height, scene) sizes of an uneven batch: fixed by the case."""
    rng = random.Random(case["size_seed"])
    scenes = [(rng.choice((3, 6, 7)), rng.choice((0, 1)), _log_int(rng, case["p_lo"], case["p_hi"])) for _ in range(case["scenes"])]
    return scenes, [(_log_int(rng, 256, 1920), _log_int(rng, 256, 1080), rng.randrange(case["scenes"])) for _ in range(case["jobs"])]


def _batch_inputs(case, seed):
    sizes, jobs = _batch_sizes(case)
    rng = random.Random(seed)
    scenes = [(N, rot, _scene(_gen(seed, 17 + i), N, P, rot, "clusters")) for i, (N, rot, P) in enumerate(sizes)]
    views = [_view(*_pose(rng), w, h, rng.random(), s) for w, h, s in jobs]
    return scenes, views, S.RasterConfig(tile_w=case["tile_w"], tile_h=case["tile_h"])


def _signs(seed, n):
    """dL/dimage of an L1 loss: +-1/n."""
    return torch.sign(_uni(_gen(seed, 5), -1.0, 1.0, n)) / n


def _image_pair(seed, views, w, h):
    """A smooth image and a noisy target of it, packed [views][3][h][w]."""
    g = _gen(seed, 7)
    low = torch.rand(views, 3, h // 8 + 2, w // 8 + 2, generator=g, device=DEV)
    img = torch.nn.functional.interpolate(low, size=(h, w), mode="bilinear", align_corners=False)
    tgt = (img + 0.1 * torch.randn(img.shape, generator=g, device=DEV)).clamp(0.0, 1.0)
    return img.reshape(-1).contiguous(), tgt.reshape(-1).contiguous()


def _moments(g, K, P):
    """Adam moments of a run under way: gradients of the scale training sees."""
    s = _log_uni(g, 1e-6, 1e-4, K, P)
    return 0.3 * s * _nrm(g, K, P), s * s


# ---------------------------------------------------------------------------------------------- one pass

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("render", "step", "graph", "autograd", "train", "batch"):
        scenes, views, cfg = _batch_inputs(case, seed) if kind == "batch" else _raster_inputs(case, seed)
        ds = [raster.DeviceScene(N, rot, p) for N, rot, p in scenes]
        if kind == "batch":
            b = raster.Batch(ds, views, cfg, [list(range(len(views)))], device=DEV)
            b.size()
            return {"kind": kind, "batch": b, "dL": [_signs(seed, r.image.numel()) for r in b.rasterizers]}
        r = raster.Rasterizer(ds, views, cfg, device=DEV)
        r.forward(check=True)
        st = {"kind": kind, "r": r}
        if kind in ("step", "graph"):
            st["dL"] = _signs(seed, r.image.numel())
        if kind == "graph":
            st["graph"] = r.capture(st["dL"])
        if kind == "autograd":
            st["params"] = [d.params.requires_grad_(True) for d in ds]
            st["dL"] = _signs(seed, r.image.numel())
        if kind == "train":
            opt = TR.Adam(ds[0], ds[0].params)
            g = _gen(seed, 11)
            opt.m[:], opt.v[:] = _moments(g, opt.K, opt.P)
            opt.step_count = 1000
            tgt = _image_pair(seed, case["views"], case["width"], case["height"])[1]
            st.update(opt=opt, loss=TR.ImageLoss(views), target=tgt, dL=torch.empty_like(r.image))
        return st
    if kind == "loss":
        views = [S.make_view(torch.eye(3).numpy(), torch.zeros(3).numpy(), case["width"], case["height"])] * case["views"]
        img, tgt = _image_pair(seed, case["views"], case["width"], case["height"])
        return {"kind": kind, "loss": TR.ImageLoss(views), "image": img, "target": tgt, "dL": torch.empty_like(img)}
    g = _gen(seed)
    act = _scene(g, case["N"], case["P"], case["rot"], "clusters")
    ds = raster.DeviceScene(case["N"], case["rot"], act)
    opt = TR.Adam(ds, act)
    opt.m[:], opt.v[:] = _moments(g, opt.K, opt.P)
    opt.step_count = 1000
    if kind == "adam":
        grad = _log_uni(g, 1e-6, 1e-4, opt.K, opt.P) * _nrm(g, opt.K, opt.P)
        noise = 1e-4 * _nrm(g, 3, opt.P) if case["noise"] else None
        return {"kind": kind, "opt": opt, "grad": grad, "noise": noise}
    rel = TR.Relocator(opt)
    row = rel.opacity_row
    dead = torch.rand(opt.P, generator=g, device=DEV) < case["dead"]
    act[row] = torch.where(dead, _uni(g, 0.0, 0.0049, opt.P), act[row].clamp(0.006, 0.999))
    opt.raw[row] = torch.logit(act[row])
    rand = torch.randint(-(1 << 63), (1 << 63) - 1, (opt.P,), generator=g, device=DEV, dtype=torch.int64)
    return {"kind": kind, "opt": opt, "rel": rel, "rand": rand, "opacity": act[row].clone()}


def run(state):
    kind = state["kind"]
    if kind == "render":
        return {"image": state["r"].forward(check=False)}
    if kind == "step":
        img = state["r"].forward(check=False)
        return {"image": img, "grads": state["r"].backward(state["dL"])}
    if kind == "graph":
        state["graph"].replay()
        return {"image": state["r"].image, "grads": state["r"].grads}
    if kind == "autograd":
        for p in state["params"]:
            p.grad = None
        img = raster.rasterize(state["r"], *state["params"])
        img.backward(state["dL"])
        return {"image": img.detach(), "grads": [p.grad for p in state["params"]]}
    if kind == "batch":
        grads = state["batch"].step(state["dL"])
        return {"image": [r.image for r in state["batch"].rasterizers], "grads": grads}
    if kind == "loss":
        return {"loss": state["loss"](state["image"], state["target"], state["dL"]), "dL": state["dL"]}
    opt = state["opt"]
    if kind == "train":
        loss = TR.train_step(state["r"], state["loss"], [opt], state["target"], state["dL"])
        return {"loss": loss, "image": state["r"].image, "dL": state["dL"], "grads": state["r"].grads, "raw": opt.raw,
                "act": opt.act, "m": opt.m, "v": opt.v}
    if kind == "adam":
        opt.step(state["grad"], state["noise"])
        return {"raw": opt.raw, "act": opt.act, "m": opt.m, "v": opt.v}
    # the opacities as the pruning pass of the trainer left them: a relocation revives the dead ones
    opt.act[state["rel"].opacity_row].copy_(state["opacity"])
    src, n = state["rel"](state["rand"])
    return {"sources": src, "n": n, "raw": opt.raw, "act": opt.act, "m": opt.m, "v": opt.v}


# ---------------------------------------------------------------------------------------------- its work

def _rows(N, rot):
    return S.params_per_primitive(N, rot)


def _pairs(P, w, h):
    """Pairs a view composites, roughly: each drawn primitive covers some hundred pixels, and a pixel saturates
    after a few tens of primitives."""
    return min(40.0 * w * h, 120.0 * P)


def _step_work(N, rot, P, views, backward):
    K = _rows(N, rot)
    pix = sum(w * h for w, h in views)
    pairs = sum(_pairs(P, w, h) for w, h in views) / (1.0 if N == 3 else 6.0)
    by = 4.0 * K * P + 12.0 * pix
    fl = 250.0 * P * len(views) + 18.0 * pairs
    if backward:
        by += 4.0 * K * P + 12.0 * pix
        fl += 500.0 * P + 48.0 * pairs
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sizes, jobs = _batch_sizes(case)
        by = fl = 0.0
        for s, (N, rot, P) in enumerate(sizes):
            b, f = _step_work(N, rot, P, [(w, h) for w, h, k in jobs if k == s], True)
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    if kind == "loss":
        n = 3.0 * case["views"] * case["width"] * case["height"]
        return {"bytes": 12.0 * n, "flops": 206.0 * n}  # image and target read, dL written; two separable window passes
    if kind in ("adam", "relocate"):
        K, P = _rows(case["N"], case["rot"]), case["P"]
        if kind == "adam":  # raw, grad, m, v read; raw, m, v, act written
            return {"bytes": 32.0 * K * P + (12.0 * P if case["noise"] else 0.0), "flops": 20.0 * K * P}
        # opacity restored and read, each dead slot's draw and its copied planes, its source's moments and every source index
        return {"bytes": 16.0 * P + case["dead"] * P * (8.0 + 32.0 * K), "flops": 4.0 * P}
    by, fl = _step_work(case["N"], case["rot"], case["P"], [(case["width"], case["height"])] * case["views"], kind != "render")
    if kind == "train":
        n, K = 3.0 * case["views"] * case["width"] * case["height"], _rows(case["N"], case["rot"])
        by += 4.0 * n + 28.0 * K * case["P"]
        fl += 206.0 * n + 20.0 * K * case["P"]
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------------------------- the pass in float64

def _rotation(rot, mode):
    if mode == 1:
        o1, o2, o3 = rot
        one = torch.ones_like(o1)
        rows = [one, -o3, o2, o3, one, -o1, -o2, o1, one]
    else:
        w, x, y, z = rot / rot.norm(dim=0, keepdim=True)
        rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z), 1 - 2 * (x * x + z * z),
                2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, -1).reshape(-1, 3, 3)


def _records(N, mode, prm, v, cfg):
    """Depth, screen mean, conic, opacity, exponent, colour of every primitive in a view (Sec. 3, 4.2-4.4), and which can be drawn."""
    C = N - 3
    off = {}
    at = 0
    for name, rows in S.plane_rows(N, mode).items():
        off[name] = prm[at:at + rows]
        at += rows
    P = prm.shape[1]
    W = torch.tensor(v.R, dtype=torch.float64, device=DEV)
    t = torch.tensor(v.t, dtype=torch.float64, device=DEV)
    mx = off["mean_x"].T
    M = _rotation(off["rot"], mode) * off["scale_x"].T[:, None, :]
    Sc = M @ M.transpose(1, 2)
    o = off["opacity"][0]
    beta = 4.0 * torch.exp(off["b"][0])
    good = torch.ones(P, dtype=torch.bool, device=DEV)
    if C:
        q = []
        if C in (1, 4):
            q.append(torch.full((P, 1), float(v.time), dtype=torch.float64, device=DEV))
        if C >= 3:
            d = mx + W.T @ t
            q.append(d / d.norm(dim=1, keepdim=True))
        delta = torch.cat(q, 1) - off["mean_q"].T
        Lqx = off["L_qx"].T.reshape(P, C, 3)
        Sqx = Lqx @ M.transpose(1, 2)
        Lq = [[off["L_q"][i * (i + 1) // 2 + j] if j <= i else None for j in range(C)] for i in range(C)]
        L, y, Z = {}, [], [None] * C  # Cholesky factor of Sigma_q by columns of scalars, L y = delta, Z = Sigma_q^-1 Sigma_qx
        for i in range(C):
            for j in range(i + 1):
                s = (Lqx[:, i] * Lqx[:, j]).sum(1) + sum(Lq[i][m] * Lq[j][m] for m in range(j + 1))
                s = s - sum(L[i, m] * L[j, m] for m in range(j))
                L[i, j] = s.sqrt() if i == j else s / L[j, j]
        for i in range(C):
            y.append((delta[:, i] - sum(L[i, m] * y[m] for m in range(i))) / L[i, i])
        Y = []
        for i in range(C):
            Y.append((Sqx[:, i] - sum(L[i, m][:, None] * Y[m] for m in range(i))) / L[i, i][:, None])
        for i in reversed(range(C)):
            Z[i] = (Y[i] - sum(L[m, i][:, None] * Z[m] for m in range(i + 1, C))) / L[i, i][:, None]
        y, Z = torch.stack(y, 1), torch.stack(Z, 1)
        bq = torch.exp(off["b"][1:]).T
        W3 = (Z * torch.clamp(bq, max=1.0)[:, :, None]).transpose(1, 2)
        M2 = W3 @ Sqx
        Sc = Sc - 0.5 * (M2 + M2.transpose(1, 2))
        x = y * y
        o = o * torch.exp((4.0 * bq * (math.log(2.0) - 2.0 * x - torch.log1p(torch.exp(-2.0 * x)))).sum(1))
        mx = mx + (W3 @ delta[:, :, None])[:, :, 0]
    tc = mx @ W.T + t
    tz = tc[:, 2]
    good = good & (tz > cfg.near) & (o >= cfg.alpha_min)
    z = torch.where(good, tz, torch.ones_like(tz))
    u, w = tc[:, 0] / z, tc[:, 1] / z
    mu = torch.stack([v.fx * u + v.cx, v.fy * w + v.cy], 1)
    lx, ly = cfg.jac_clip * 0.5 * v.width / v.fx, cfg.jac_clip * 0.5 * v.height / v.fy
    zero = torch.zeros_like(z)
    J = torch.stack([v.fx / z, zero, -v.fx * u.clamp(-lx, lx) / z, zero, v.fy / z, -v.fy * w.clamp(-ly, ly) / z], 1).reshape(P, 2, 3)
    T = J @ W
    cov = T @ Sc @ T.transpose(1, 2)
    s00, s01, s11 = cov[:, 0, 0] + cfg.eps2d, cov[:, 0, 1], cov[:, 1, 1] + cfg.eps2d
    det = s00 * s11 - s01 * s01
    good = good & (det > 0)
    det = torch.where(good, det, torch.ones_like(det))
    rec = torch.stack([mu[:, 0], mu[:, 1], s11 / det, -s01 / det, s00 / det, o, beta, off["rgb"][0], off["rgb"][1], off["rgb"][2]], 1)
    with torch.no_grad():  # boxes of the pixels with alpha >= alpha_min, widened by a pixel
        rc = torch.where(good, 1.0 - (cfg.alpha_min / o.clamp(min=1e-30)) ** (1.0 / beta), zero)
        rc = rc.clamp(0.0, 1.0)
        ex, ey = (rc * s00).clamp(min=0).sqrt() + 1.0, (rc * s11).clamp(min=0).sqrt() + 1.0
        box = torch.stack([mu[:, 0] - ex, mu[:, 0] + ex, mu[:, 1] - ey, mu[:, 1] + ey], 1)
        good = good & (box[:, 1] >= 0) & (box[:, 0] <= v.width) & (box[:, 3] >= 0) & (box[:, 2] <= v.height)
    return rec, tz, box, good


def _composite(rec, px, py, cfg):
    """Colours [pixels, 3] of depth-ordered records (Sec. 3)."""
    dx, dy = px[:, None] - rec[None, :, 0], py[:, None] - rec[None, :, 1]
    r = rec[:, 2] * dx * dx + 2.0 * rec[:, 3] * dx * dy + rec[:, 4] * dy * dy
    inside = r < 1.0
    alpha = rec[:, 5] * torch.where(inside, 1.0 - r, torch.full_like(r, 0.5)) ** rec[:, 6]
    alpha = alpha.clamp(max=cfg.alpha_max)
    a = torch.where(inside & (alpha >= cfg.alpha_min), alpha, torch.zeros_like(alpha))
    with torch.no_grad():
        alive = torch.cumprod(1.0 - a, 1) >= cfg.T_min
    a = torch.where(alive, a, torch.zeros_like(a))
    T = torch.cumprod(1.0 - a, 1)
    before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    return (a * before) @ rec[:, 7:10] + T[:, -1:] * torch.tensor(cfg.bg, dtype=torch.float64, device=DEV)


def _exact_raster(scenes, views, cfg, dL=None, side=64):
    """Packed image and, with dL (packed; or a function of the image), the gradients of every scene."""
    images, saved = [], []
    prms = [p.double().detach().requires_grad_(True) for _, _, p in scenes]
    for v in views:
        N, mode, _ = scenes[v.scene_id]
        with torch.enable_grad():
            rec, tz, box, good = _records(N, mode, prms[v.scene_id], v, cfg)
        keep = good.nonzero()[:, 0]
        keep = keep[torch.argsort(tz.detach()[keep].float(), stable=True)]
        leaf, bx = rec.detach()[keep], box[keep]
        img = torch.zeros(3, v.height, v.width, dtype=torch.float64, device=DEV)
        img += torch.tensor(cfg.bg, dtype=torch.float64, device=DEV)[:, None, None]
        blocks = []
        todo = [(x, y, side) for y in range(0, v.height, side) for x in range(0, v.width, side)]
        while todo:
            x0, y0, s = todo.pop()
            x1, y1 = min(v.width, x0 + s), min(v.height, y0 + s)
            if x0 >= x1 or y0 >= y1:
                continue
            hit = ((bx[:, 1] >= x0) & (bx[:, 0] <= x1) & (bx[:, 3] >= y0) & (bx[:, 2] <= y1)).nonzero()[:, 0]
            if not hit.numel():
                continue
            if hit.numel() * s * s > 4_000_000 and s > 8:
                h = s // 2
                todo += [(x0, y0, h), (x0 + h, y0, h), (x0, y0 + h, h), (x0 + h, y0 + h, h)]
                continue
            gy, gx = torch.meshgrid(torch.arange(y0, y1, device=DEV), torch.arange(x0, x1, device=DEV), indexing="ij")
            px, py = gx.reshape(-1).double() + 0.5, gy.reshape(-1).double() + 0.5
            with torch.no_grad():
                img[:, y0:y1, x0:x1] = _composite(leaf[hit], px, py, cfg).T.reshape(3, y1 - y0, x1 - x0)
            blocks.append((x0, y0, x1, y1, px, py, hit))
        images.append(img)
        saved.append((rec, keep, leaf, blocks))
    image = torch.cat([i.reshape(-1) for i in images])
    if dL is None:
        return image, None, None
    dL = dL(image) if callable(dL) else dL.double()
    at = 0
    for v, (rec, keep, leaf, blocks) in zip(views, saved):
        n = 3 * v.width * v.height
        gi = dL[at:at + n].view(3, v.height, v.width)
        at += n
        g = torch.zeros_like(leaf)
        for x0, y0, x1, y1, px, py, hit in blocks:
            with torch.enable_grad():
                part = leaf[hit].requires_grad_(True)
                col = _composite(part, px, py, cfg)
            g.index_add_(0, hit, torch.autograd.grad(col, part, gi[:, y0:y1, x0:x1].reshape(3, -1).T)[0])
        full = torch.zeros(rec.shape, dtype=torch.float64, device=DEV)
        full[keep] = g
        rec.backward(full)
    return image, [p.grad if p.grad is not None else torch.zeros_like(p) for p in prms], dL


def _exact_loss(img, tgt, views, lam=TR.LAMBDA_SSIM):
    """[total, per view] and dL/dimage of (1 - lam) L1 + lam (1 - SSIM), 11 x 11 window of sigma 1.5."""
    k = torch.exp(-((torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2) / (2 * 1.5 * 1.5))
    k = k / k.sum()

    def blur(x):
        x = torch.nn.functional.pad(x, (5, 5, 5, 5))
        H, W = x.shape[1] - 10, x.shape[2] - 10
        x = sum(k[i] * x[:, :, i:i + W] for i in range(11))
        return sum(k[i] * x[:, i:i + H] for i in range(11))

    losses, at = [], 0
    with torch.enable_grad():
        x = img.double().detach().requires_grad_(True)
        for w, h in views:
            a, b = (z[at:at + 3 * w * h].view(3, h, w) for z in (x, tgt.double()))
            at += 3 * w * h
            ma, mb = blur(a), blur(b)
            va, vb, ab = blur(a * a) - ma * ma, blur(b * b) - mb * mb, blur(a * b) - ma * mb
            s = ((2 * ma * mb + 1e-4) * (2 * ab + 9e-4)) / ((ma * ma + mb * mb + 1e-4) * (va + vb + 9e-4))
            losses.append((1 - lam) * (a - b).abs().mean() + lam * (1 - s.mean()))
        total = torch.stack(losses).mean()
        g, = torch.autograd.grad(total, x)
    return torch.stack([total, *losses]).detach(), g


def _exact_adam(opt, raw, m, v, grad, noise):
    """(raw, act, m, v) after the step the optimiser takes next."""
    tc = opt.tc
    raw, m, v, g = (x.double() for x in (raw, m, v, grad))
    t = opt.step_count + 1

    def act(x):
        y = x.clone()
        for k, (_, a, _, _) in enumerate(opt.table):
            y[k] = torch.sigmoid(x[k]) if a == ACT_SIGMOID else torch.exp(x[k]) if a == ACT_EXP else x[k]
        return y

    a0 = act(raw)
    col = lambda j: torch.tensor([float(p[j]) for p in opt.table], dtype=torch.float64, device=DEV)[:, None]  # noqa: E731
    g = g + col(2) * torch.sign(a0)
    for k, (_, a, _, _) in enumerate(opt.table):
        g[k] = g[k] * (a0[k] * (1 - a0[k]) if a == ACT_SIGMOID else a0[k] if a == ACT_EXP else 1.0)
    m = tc.beta1 * m + (1 - tc.beta1) * g
    v = tc.beta2 * v + (1 - tc.beta2) * g * g
    raw = raw - col(0) * (m / (1 - tc.beta1 ** t)) / ((v / (1 - tc.beta2 ** t)).sqrt() + tc.eps)
    if noise is not None:
        for k, (_, _, _, row) in enumerate(opt.table):
            if row >= 0:
                raw[k] = raw[k] + tc.lambda_eps * noise[row].double()
    return raw, act(raw), m, v


def exact(case, seed):
    kind = case["kind"]
    if kind in ("render", "step", "graph", "autograd"):
        scenes, views, cfg = _raster_inputs(case, seed)
        dL = None if kind == "render" else _signs(seed, 3 * sum(v.width * v.height for v in views))
        img, grads, _ = _exact_raster(scenes, views, cfg, dL)
        return {"image": img} if grads is None else {"image": img, "grads": grads}
    if kind == "batch":
        return None  # some dozen views of large scenes: over the time there is for float64
    st = prepare(case, seed)
    if kind == "loss":
        loss, g = _exact_loss(st["image"], st["target"], [(case["width"], case["height"])] * case["views"])
        return {"loss": loss, "dL": g}
    opt = st["opt"]
    if kind == "adam":
        return dict(zip(("raw", "act", "m", "v"), _exact_adam(opt, opt.raw, opt.m, opt.v, st["grad"], st["noise"])))
    if kind == "train":
        scenes, views, cfg = _raster_inputs(case, seed)
        got = {}

        def loss_of(img):
            got["loss"], g = _exact_loss(img, st["target"], [(v.width, v.height) for v in views])
            return g

        img, grads, g = _exact_raster(scenes, views, cfg, loss_of)
        new = _exact_adam(opt, opt.raw, opt.m, opt.v, grads[0], None)
        return {"loss": got["loss"], "image": img, "dL": g, "grads": grads, **dict(zip(("raw", "act", "m", "v"), new))}
    row, P = st["rel"].opacity_row, opt.P
    o = st["opacity"]
    live = o > TR.DEAD_THRESHOLD
    cum = torch.cumsum(torch.where(live, (o.double() * 16777216.0).floor().long(), torch.zeros(P, dtype=torch.int64, device=DEV)), 0)
    total = int(cum[-1])
    half = 1 << 32  # rand as an unsigned 64-bit integer, modulo the total weight, by halves
    hi, lo = (st["rand"] >> 32) & (half - 1), st["rand"] & (half - 1)
    rem = hi % total
    for _ in range(32):
        rem = (rem * 2) % total
    draw_ = (rem + lo % total) % total
    src = torch.searchsorted(cum, draw_, right=True)
    src = torch.where(live, torch.full_like(src, -1), src)
    dead = (~live).nonzero()[:, 0]
    from_ = src[dead]
    n = torch.zeros(P, dtype=torch.int64, device=DEV).index_add_(0, from_, torch.ones_like(from_))
    act, raw = opt.act.double(), opt.raw.double()
    act[row] = o.double()
    new = 1.0 - (1.0 - act[row]) ** (1.0 / (n + 1).double())
    touched = n > 0
    act[:, dead], raw[:, dead] = act[:, from_], raw[:, from_]
    act[row] = torch.where(touched, new, o.double())
    raw[row] = torch.where(touched, torch.logit(new), raw[row])
    act[row, dead], raw[row, dead] = new[from_], torch.logit(new[from_])
    m, v = opt.m.double(), opt.v.double()
    both = torch.cat([dead, touched.nonzero()[:, 0]])
    m[:, both] = 0.0
    v[:, both] = 0.0
    return {"sources": src.int(), "n": torch.tensor([dead.numel()]), "raw": raw, "act": act, "m": m, "v": v}

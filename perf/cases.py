"""What is timed of this framework, case by case, through its public entry points.

A case is a dict of plain values; ``listed()`` gives the standing ones and
``draw()`` more of the same ranges.  ``prepare()`` makes what a user's program
has in hand before the call (a context with its map loaded, the query images
on the GPU, poses), ``run()`` makes the call, ``work()`` counts what the path
cannot do without and ``exact()`` restates the result in 64 bits with plain
torch.

Maps are the seeded synthetic scenes of ``scenegen``.  A map is fixed by its
kind, size and degree, as a deployment has one map that many queries meet; what
the seed draws is the queries: hidden and coarse poses, image noise, visiting
orders, pixel pairs, training views, network inputs.  The contexts that hold
maps are kept between states for the same reason.

Query images and training targets come from the renderer below (FP64, plain
torch), not from the framework.

Outputs carry the type that the path computes them in: what is rendered, and
what is formed from renders (NCC scores, their pose gradient, the training
loss), is FP32 work that the C ABI hands out as double, and is returned as
float32; poses and the PnP solution are FP64 throughout and stay float64.
"""
from __future__ import annotations

import collections
import functools
import math

import numpy as np
import torch

import scenegen as sg
from paper_2403_11367_gb300 import reloc as R

DEV = "cuda:0"
STORES = {"fp32": (R.FP32, torch.float32), "fp16": (R.FP16, torch.float16), "bf16": (R.BF16, torch.bfloat16)}
BLOCK = {"street": 20.0, "box": 5.0}       # 2D voxel edge, metres

# the driving camera and map of the benchmark
STREET = {"map": "street", "n": 2_000_000, "w": 1408, "h": 376, "focal": 552.0, "radius": 40.0}
BOX = {"map": "box", "n": 10_000, "w": 352, "h": 94, "focal": 138.0, "radius": 30.0}
GRID64 = {"nx": 4, "ny": 4, "nyaw": 4, "step_xy": 0.5, "step_yaw": 2.0}


def listed():
    return [
        # a preview or a unit-sized render of a small map: launches and latency
        {"name": "render_box", "path": "render", **BOX, "sh": 0, "store": "fp32", "views": 1},
        # one step of the refinement loop: RGB, depth and alpha of one driving view
        {"name": "render_street", "path": "render", **STREET, "sh": 3, "store": "fp32", "views": 1},
        # relocalization in a small map with a small odd grid
        {"name": "localize_box", "path": "localize", **BOX, "sh": 0, "store": "fp32", "nx": 3, "ny": 3, "nyaw": 2,
         "step_xy": 0.5, "step_yaw": 3.0},
        # the headline: 64 candidates of one driving query, winner exported
        {"name": "localize_street", "path": "localize", **STREET, "sh": 3, "store": "fp32", **GRID64},
        # a server's batch of uneven queries (8 to 128 candidates, 15 to 95 m) on a map stored in 16 bits
        {"name": "batch_street", "path": "batch", **STREET, "sh": 3, "store": "bf16", "queries": 8},
        # the same with the learned proposal: the top 8 cells of each query, the full sweep where it is unsure
        {"name": "serve_learned", "path": "serve", **STREET, "sh": 3, "store": "bf16", "queries": 32, "top_k": 8,
         "margin": 0.052},
        # the paper's random search: 20% of 8100 cells over (-15, 15) m and a full turn, batches of 64
        {"name": "search_street", "path": "search", **STREET, "sh": 3, "store": "fp16", "nx": 15, "ny": 15,
         "nyaw": 36, "step_xy": 2.0, "step_yaw": 10.0, "fraction": 0.2, "batch": 64, "ncc_stop": 0.8},
        # one gradient evaluation of direct pose ascent on NCC
        {"name": "pose_grad", "path": "grad", **STREET, "sh": 0, "store": "fp32", "views": 1},
        # the PnP solve of the refinement, some 7400 pixel pairs
        {"name": "refine_pnp", "path": "pnp", **STREET, "sh": 0, "store": "fp32", "step": 8, "noise": 0.5,
         "outliers": 0.1},
        # loss and gradient of one map-training step over a 16-view driving sequence
        {"name": "train_street", "path": "train", **STREET, "sh": 0, "store": "fp32", "views": 16},
        # one training step of the proposal network at its training batch
        {"name": "proposal_train", "path": "proposal", "batch": 256},
        # the dense contraction of the proposal's first full layer at a large batch
        {"name": "gemm_fc1", "path": "gemm", "m": 8192, "nn": 1024, "k": 1536, "relu": True, "split": 1},
    ]


def _between(rng, lo, hi):
    """A whole number of [lo, hi], spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["render", "render", "localize", "localize", "localize", "batch", "serve", "search", "grad",
                       "pnp", "train", "proposal", "gemm", "gemm"])
    if path == "proposal":
        return {"path": path, "batch": 64 * _between(rng, 1, 8)}
    if path == "gemm":
        return {"path": path, "m": _between(rng, 48, 8192), "nn": _between(rng, 33, 2048),
                "k": 64 * _between(rng, 2, 48), "relu": rng.random() < 0.5, "split": 1}
    if path == "serve":
        return {"path": path, **STREET, "sh": 3, "store": rng.choice(["fp32", "bf16"]),
                "queries": _between(rng, 1, 32), "top_k": rng.randint(4, 16), "margin": 0.052}
    small = path in ("render", "localize") and rng.random() < 0.3
    if small:
        w = rng.randint(160, 400)
        case = {"path": path, "map": "box", "n": _between(rng, 1000, 30_000), "w": w, "h": rng.randint(60, 140),
                "focal": round(0.39 * w, 1), "radius": 30.0}
    else:
        w = rng.randint(600, 1408)
        case = {"path": path, "map": "street", "n": _between(rng, 100_000, 2_000_000), "w": w,
                "h": rng.randint(160, 376), "focal": round(0.39 * w, 1), "radius": round(rng.uniform(25.0, 60.0), 1)}
    flat = path in ("grad", "pnp", "train")
    case["sh"] = 0 if flat else rng.choice([0, 1, 2, 3])
    case["store"] = "fp32" if flat else rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if path in ("render", "grad"):
        case["views"] = _between(rng, 1, 16)
    if path == "train":
        case["views"] = rng.randint(2, 16)
    if path == "localize":
        case.update(nx=rng.randint(1, 5), ny=rng.randint(1, 5), nyaw=rng.randint(2, 5),
                    step_xy=round(rng.uniform(0.25, 1.0), 2), step_yaw=round(rng.uniform(1.0, 4.0), 1))
    if path == "batch":
        case["queries"] = rng.randint(2, 8)
    if path == "search":
        case.update(nx=rng.randint(5, 15), ny=rng.randint(5, 15), nyaw=rng.randint(12, 36), step_xy=2.0, step_yaw=10.0,
                    fraction=round(rng.uniform(0.05, 0.2), 3), batch=_between(rng, 16, 128), ncc_stop=0.8)
    if path == "pnp":
        case.update(step=rng.randint(4, 24), noise=0.5, outliers=round(rng.uniform(0.0, 0.25), 2))
    return case


# ---------------------------------------------------------------------------
# maps, contexts, inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _gaussians(kind, n, sh):
    if kind == "box":
        return sg.tiny_scene(n=n).gaussians
    return sg.street_gaussians(n, seed=11, sh_degree=sh)


def _noisy(g):
    """The start map of a training run: the true one with noise on opacity and colour."""
    r = sg.Rng(17)
    return sg.Gaussians(g.mean, g.scale, g.quat,
                        np.clip(g.opacity + r.normal(g.n, 0.0, 0.1), 0.02, 0.98).astype(np.float32),
                        np.clip(g.sh + r.normal(g.sh.size, 0.0, 0.1).reshape(g.sh.shape), 0.0, 1.0).astype(np.float32),
                        g.sh_degree)


def _map(case):
    g = _gaussians(case["map"], case["n"], 0 if case["map"] == "box" else case["sh"])
    return _noisy(g) if case["path"] == "train" else g


_CONTEXTS = collections.OrderedDict()


def _context(case):
    """The program's context for this map (kept, as a server keeps it)."""
    role = case["path"] if case["path"] in ("train", "batch", "serve") else "any"
    key = (case["map"], case["n"], case["sh"], case["store"], role, case.get("top_k"), case.get("margin"))
    if key not in _CONTEXTS:
        ctx = R.Context(R.reloc_default_config(block_size=BLOCK[case["map"]]))
        ctx.load_map(_map(case), STORES[case["store"]][0])
        if role in ("batch", "serve"):
            ctx.set_batch_options(use_graph=True, mem_budget=24 << 30)
        if role == "serve":
            ctx.proposal_init(0)
            ctx.proposal_set_params(np.fromfile("paper_2403_11367_gb300/weights/proposal_street.bin", dtype="<f4"))
            ctx.set_proposal(True, case["top_k"], case["margin"])
        _CONTEXTS[key] = ctx
        while len(_CONTEXTS) > 6:
            _CONTEXTS.popitem(last=False)
    _CONTEXTS.move_to_end(key)
    return _CONTEXTS[key]


def _camera(case):
    return sg.Camera(case["w"], case["h"], case["focal"], case["focal"], case["w"] / 2.0, case["h"] / 2.0)


def _box_poses(n, seed):
    """(hidden, coarse) pose tuples in front of the box, within 1 m and 5 degrees of its seed pose."""
    r = sg.Rng(seed)
    o = np.stack([r.uniform(2 * n, -1, 1), r.uniform(2 * n, -1, 1), r.uniform(2 * n, -math.radians(5), math.radians(5))], 1)
    p = [(float(a), -14.0 + float(b), 2.0, math.pi / 2 + float(c)) for a, b, c in o]
    return p[:n], p[n:]


def _poses(case, n, seed):
    return _box_poses(n, seed) if case["map"] == "box" else sg.street_queries(n, seed=seed)


def _noise(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return 0.02 * torch.randn((3, case["h"], case["w"]), generator=g, device=DEV)


def _query_image(case, hidden, radius, seed):
    """The camera's image at the hidden pose: the true map rendered there, with sensor noise."""
    s = _subset(case, _gaussians(case["map"], case["n"], 0 if case["map"] == "box" else case["sh"]), "fp32", hidden,
                radius)
    rgb = _render64(s, _wp(hidden), _camera(case))[0]
    return (rgb.float() + _noise(case, seed)).contiguous()


def _wp(p):
    return sg.pose_from_xyz_yaw(*p)


def _inputs(case, seed):
    """Everything that the seed decides, as both prepare() and exact() take it."""
    path = case["path"]
    base = 7919 * (seed + 1)
    if path == "gemm":
        g = torch.Generator(device=DEV)
        g.manual_seed(base)
        return {"a": torch.randn((case["m"], case["k"]), generator=g, device=DEV).to(torch.bfloat16),
                "b": (torch.randn((case["nn"], case["k"]), generator=g, device=DEV) / math.sqrt(case["k"])).to(torch.bfloat16),
                "bias": 0.1 * torch.randn((case["nn"],), generator=g, device=DEV)}
    if path == "proposal":
        g = torch.Generator(device=DEV)
        g.manual_seed(base)
        b = case["batch"]
        x = torch.rand((b, R.PROPOSAL_H, R.PROPOSAL_W, 2), generator=g, device=DEV).to(torch.bfloat16)
        y = torch.randint(0, R.PROPOSAL_CLASSES, (b,), generator=g, device=DEV, dtype=torch.int32)
        parts = []
        for shape in _PROPOSAL_SHAPES:
            n = math.prod(shape)
            std = math.sqrt(2.0 / math.prod(shape[1:])) if len(shape) > 1 else 0.01
            parts.append(std * torch.randn((n,), generator=g, device=DEV))
        return {"x": x, "y": y, "params": torch.cat(parts).cpu().numpy()}
    if path in ("render", "grad"):
        hidden, coarse = _poses(case, case["views"] + 1, base)
        h = hidden[0]
        # the views of one call look at one place: the first coarse pose and steps around it
        r = sg.Rng(base + 1)
        views = [(coarse[0][0] + d[0], coarse[0][1] + d[1], coarse[0][2], coarse[0][3] + math.radians(3) * d[2])
                 for d in r.uniform(3 * case["views"], -1, 1).reshape(-1, 3)]
        out = {"poses": np.stack([_wp(v) for v in views]), "at": coarse[0]}
        if path == "grad":
            out["query"] = _query_image(case, h, case["radius"], base)
        return out
    if path == "localize":
        hidden, coarse = _poses(case, 1, base)
        return {"query": _query_image(case, hidden[0], case["radius"], base), "coarse": coarse[0]}
    if path == "search":
        hidden, _ = _poses(case, 1, base)
        r = sg.Rng(base + 1)
        h, d = hidden[0], [float(r.uniform(1, -m, m)[0]) for m in (10.0, 10.0, math.pi / 2)]
        return {"query": _query_image(case, h, case["radius"], base),
                "coarse": (h[0] + d[0], h[1] + d[1], h[2], h[3] + d[2]), "seed": base}
    if path in ("batch", "serve"):
        hidden, coarse = _poses(case, case["queries"], base)
        r = sg.Rng(case["queries"])                # the grids and radii are the case's, the poses the seed's
        qs = []
        for i in range(case["queries"]):
            grid, radius = (4, 4, 4, 0.5, 2.0), case["radius"]
            if path == "batch":
                u = r.uniform(4)
                grid = (2 + int(3 * u[0]), 2 + int(3 * u[1]), 2 + int(7 * u[2]), 0.5, 2.0)
                radius = 15.0 + 80.0 * float(u[3])
            qs.append((_query_image(case, hidden[i], radius, base + i), coarse[i], radius, grid))
        return {"queries": qs}
    if path == "pnp":
        hidden, coarse = _poses(case, 1, base)
        s = _subset(case, _map(case), "fp32", coarse[0], case["radius"])
        cam = _camera(case)
        _, depth, alpha = _render64(s, _wp(coarse[0]), cam, True)
        depth, alpha = depth.float(), alpha.float()
        return {"pose": _wp(coarse[0]), "depth": depth.contiguous(), "alpha": alpha.contiguous(),
                "pairs": _pixel_pairs(case, _wp(coarse[0]), _wp(hidden[0]), cam, depth, alpha, base)}
    if path == "train":
        hidden, _ = _poses(case, 1, base)
        x, y, z, yaw = hidden[0]
        v = case["views"]
        views = [(x + k * math.cos(yaw), y + k * math.sin(yaw), z, yaw) for k in range(v)]
        mid, radius = (x + 0.5 * v * math.cos(yaw), y + 0.5 * v * math.sin(yaw)), case["radius"] + v / 2
        true = _subset(case, _gaussians(case["map"], case["n"], case["sh"]), "fp32", mid, radius)
        targets = torch.stack([_render64(true, _wp(p), _camera(case))[0].float() for p in views])
        return {"poses": np.stack([_wp(p) for p in views]), "mid": mid, "radius": radius, "targets": targets.contiguous()}
    raise ValueError(path)


def _pixel_pairs(case, w_render, w_query, cam, depth, alpha, seed):
    """A matcher's output: pixels of the render and where their points lie in the query, with noise and outliers."""
    rs = np.random.RandomState(seed % (1 << 31))
    st, H, W = case["step"], cam.height, cam.width
    d, a = depth.cpu().numpy().astype(np.float64), alpha.cpu().numpy().astype(np.float64)
    ys, xs = (m.ravel() for m in np.meshgrid(np.arange(st // 2, H - 1, st), np.arange(st // 2, W - 1, st), indexing="ij"))
    keep = a[ys, xs] >= 0.95
    ys, xs = ys[keep], xs[keep]
    z, u, v = d[ys, xs] / a[ys, xs], xs + 0.5, ys + 0.5
    pc = np.stack([z * (u - cam.cx) / cam.fx, z * (v - cam.cy) / cam.fy, z], 1)
    p = (pc - w_render[:3, 3]) @ w_render[:3, :3] @ w_query[:3, :3].T + w_query[:3, 3]
    with np.errstate(divide="ignore", invalid="ignore"):
        q = np.stack([cam.fx * p[:, 0] / p[:, 2] + cam.cx, cam.fy * p[:, 1] / p[:, 2] + cam.cy], 1)
    q += case["noise"] * rs.randn(*q.shape)
    out = rs.permutation(len(q))[:int(case["outliers"] * len(q))]
    q[out] = rs.rand(len(out), 2) * (W, H)
    ok = (p[:, 2] > 0.1) & (q[:, 0] >= 0) & (q[:, 0] < W) & (q[:, 1] >= 0) & (q[:, 1] < H)
    return torch.tensor(np.stack([u, v, q[:, 0], q[:, 1]], 1)[ok].astype(np.float32), device=DEV)


def prepare(case, seed):
    s = _inputs(case, seed)
    path = case["path"]
    s["path"], s["case"] = path, case
    if path == "gemm":
        s["ctx"] = R.Context()
        s["out"] = torch.empty((case["m"], case["nn"]), device=DEV)
        return s
    if path == "proposal":
        s["ctx"] = R.Context()
        s["ctx"].proposal_init(0)
        s["ctx"].proposal_set_params(s["params"])
        return s
    ctx = s["ctx"] = _context(case)
    s["cam"] = _camera(case)
    H, W = case["h"], case["w"]
    if path in ("render", "grad"):
        s["runs"] = ctx.select_block(s["at"][0], s["at"][1], case["radius"])[0]
        if path == "render":
            v = case["views"]
            s["rgb"], s["depth"], s["alpha"] = (torch.empty((v, c, H, W) if c else (v, H, W), device=DEV) for c in (3, 0, 0))
    if path in ("localize", "search"):
        s["pose"], s["grid"] = _wp(s["coarse"]), _grid(case)
        s["rgb"], s["depth"], s["alpha"] = (torch.empty((c, H, W) if c else (H, W), device=DEV) for c in (3, 0, 0))
    if path in ("batch", "serve"):
        s["list"] = [(img, _wp(p), radius, grid) for img, p, radius, grid in s["queries"]]
        n = case["queries"]
        s["rgb"], s["depth"] = torch.empty((n, 3, H, W), device=DEV), torch.empty((n, H, W), device=DEV)
    if path == "train":
        s["runs"] = ctx.select_block(s["mid"][0], s["mid"][1], s["radius"])[0]
        s["grad"] = torch.empty((14, ctx.n), device=DEV)
    return s


def _f32(x):
    return np.asarray(x, np.float32)


def _winner(res):
    return {"best": int(res.best_index), "score": _f32(res.best_score), "pose": np.array(res.best_pose).reshape(4, 4),
            "n_gauss": int(res.n_gauss), "n_scored": int(res.n_scored)}


def run(s):
    path, ctx, case = s["path"], s["ctx"], s["case"]
    if path == "gemm":
        ctx.gemm_bf16(s["a"], s["b"], s["out"], bias=s["bias"], relu=case["relu"], split_k=case["split"])
        return s["out"]
    if path == "proposal":
        loss = ctx.proposal_train_step(s["x"], s["y"], 1e-4)
        return {"loss": _f32(loss), "grads": ctx.proposal_get(1)}
    cam = s["cam"]
    if path == "render":
        ctx.render(s["runs"], s["poses"], cam, rgb=s["rgb"], depth=s["depth"], alpha=s["alpha"])
        return {"rgb": s["rgb"], "depth": s["depth"], "alpha": s["alpha"]}
    if path == "grad":
        sc, gr = ctx.score_grad(s["runs"], s["poses"], cam, s["query"])
        return {"scores": _f32(sc), "grads": _f32(gr)}
    if path == "localize":
        res, sc = ctx.localize(s["query"], s["pose"], case["radius"], s["grid"], cam, best_rgb=s["rgb"],
                               best_depth=s["depth"], best_alpha=s["alpha"])
        return {**_winner(res), "scores": _f32(sc), "rgb": s["rgb"], "depth": s["depth"], "alpha": s["alpha"]}
    if path == "search":
        res, sc = ctx.localize_random(s["query"], s["pose"], case["radius"], s["grid"], cam, fraction=case["fraction"],
                                      ncc_stop=case["ncc_stop"], batch=case["batch"], seed=s["seed"],
                                      best_rgb=s["rgb"], best_depth=s["depth"], best_alpha=s["alpha"])
        return {**_winner(res), "scores": _f32(sc), "rgb": s["rgb"], "depth": s["depth"], "alpha": s["alpha"]}
    if path in ("batch", "serve"):
        # one array per field over the queries; the scores of all queries end to end
        res, sc = ctx.localize_batch(s["list"], cam, best_rgb=s["rgb"], best_depth=s["depth"])
        w = [_winner(r) for r in res]
        return {**{k: np.stack([np.asarray(x[k]) for x in w]) for k in w[0]}, "scores": _f32(np.concatenate(sc)),
                "rgb": s["rgb"], "depth": s["depth"]}
    if path == "pnp":
        r = ctx.refine_pnp(s["pose"], cam, s["depth"], s["alpha"], s["pairs"])
        return {"pose": np.array(r.pose).reshape(4, 4), "rms_px": float(r.rms_px), "cost": float(r.cost),
                "n_used": int(r.n_used)}
    if path == "train":
        loss = ctx.train_grad(s["runs"], s["poses"], cam, s["targets"], s["grad"])
        return {"loss": _f32(loss), "grad": s["grad"]}
    raise ValueError(path)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the selected Gaussians' attributes once, images once.  Operations
    of a rendered view: 22 for each (pixel, Gaussian) pair whose footprint holds
    the pixel up to the pixel's stop (the benchmark's count), some 54 a pixel on
    the 2M-Gaussian street and 31 on the 10k box by the oracle's counts, fewer
    in proportion on thinner maps; a gradient costs twice its forward."""
    path = case["path"]
    if path == "gemm":
        m, n, k = case["m"], case["nn"], case["k"]
        return {"bytes": 2 * (m * k + n * k) + 4 * (n + m * n), "flops": 2 * m * n * k}
    if path == "proposal":
        convs = [(2, 32, 24, 88), (32, 64, 12, 44), (64, 64, 6, 22), (64, 128, 3, 11), (128, 128, 2, 6)]
        fwd = [2 * h * w * co * 9 * ci for ci, co, h, w in convs] + [2 * 1536 * 1024, 2 * 1024 * 64]
        # input, parameters with their moments read and written, gradients out
        return {"bytes": case["batch"] * (47 * 176 * 2 * 2 + 4) + R.PROPOSAL_PARAMS * 4 * 7,
                "flops": case["batch"] * (2 * sum(fwd) + sum(fwd[1:]))}
    hw = case["h"] * case["w"]
    if path == "pnp":
        n = hw // case["step"] ** 2
        # each of some 5 iterations: two passes over the pairs, about 150 operations a pair
        return {"bytes": n * (16 + 8 * 4), "flops": n * 5 * 2 * 150}

    def subset(radius, ahead=0.0):
        if case["map"] == "box":
            return case["n"]
        return case["n"] * min(1.0, 2 * (radius + ahead) / sg.STREET_LENGTH)

    if case["map"] == "box":
        per_pixel = 31 * case["n"] / 10_000
    else:
        per_pixel = 54 * case["n"] / 2_000_000
    attr = 12 + (4 if case["store"] == "fp32" else 2) * (8 + 3 * (case["sh"] + 1) ** 2)
    pair = 22 * per_pixel * hw
    img = 4 * hw
    if path == "render":
        v = case["views"]
        return {"bytes": subset(case["radius"]) * attr + v * 5 * img, "flops": v * pair}
    if path == "grad":
        v = case["views"]
        return {"bytes": subset(case["radius"]) * attr + 3 * img, "flops": 3 * v * pair}
    if path == "train":
        v = case["views"]
        s = subset(case["radius"], v / 2)
        return {"bytes": s * attr + 14 * 4 * case["n"] + v * 3 * img, "flops": 3 * v * pair}
    if path == "localize":
        cells = case["nx"] * case["ny"] * case["nyaw"]
    elif path == "search":
        cells = math.ceil(case["fraction"] * case["nx"] * case["ny"] * case["nyaw"])
    elif path == "batch":
        # grids of 2..4 x 2..4 x 2..8 cells, radii 15..95 m: 45 cells and 55 m on average
        q = case["queries"]
        return {"bytes": q * (subset(55.0) * attr + 7 * img), "flops": q * 46 * pair}
    else:
        q = case["queries"]
        return {"bytes": q * (subset(case["radius"]) * attr + 7 * img), "flops": q * (case["top_k"] + 2) * pair}
    # the query in, the winner's five planes out (and rendered once more)
    return {"bytes": subset(case["radius"]) * attr + 8 * img, "flops": (cells + 1) * pair}


# ---------------------------------------------------------------------------
# 64-bit restatement in plain torch
# ---------------------------------------------------------------------------

NEAR, FOV, EPS2D, A_MIN, A_MAX, T_MIN, CUT = 0.2, 1.3, 0.3, 1.0 / 255.0, 0.99, 1e-4, 3.0
EXACT_VIEWS = 200                          # candidate views that exact() renders at most


@functools.lru_cache(maxsize=2)
def _means_on_gpu(kind, n, sh):
    return torch.from_numpy(_gaussians(kind, n, sh).mean).to(DEV)


def _subset(case, g, store, at, radius):
    """The Gaussians of the 2D voxels whose centre lies within `radius` of `at`, block by
    block, as FP64 tensors of the values that the given storage holds."""
    block = BLOCK[case["map"]]
    m = _means_on_gpu(case["map"], case["n"], 0 if case["map"] == "box" else case["sh"])
    b = torch.floor(m[:, :2].double() / block)
    c = (b + 0.5) * block
    idx = torch.nonzero(torch.hypot(c[:, 0] - at[0], c[:, 1] - at[1]) <= radius)[:, 0]
    key = b[idx, 0] * 1e6 + b[idx, 1]
    idx = idx[torch.sort(key, stable=True).indices]
    host = idx.cpu().numpy()

    def up(a, rounded=True):
        t = torch.from_numpy(a[host]).to(DEV)
        return (t.to(STORES[store][1]) if rounded else t).double()
    return {"mean": up(g.mean, False), "scale": up(g.scale), "quat": up(g.quat), "opacity": up(g.opacity),
            "sh": up(g.sh), "deg": g.sh_degree, "index": idx}


def _sh_basis(deg, d):
    """Real orthonormal spherical harmonics (Condon-Shortley phase) of unit directions [n][3]."""
    re, im = [torch.ones_like(d[:, 0])], [torch.zeros_like(d[:, 0])]
    for _ in range(deg):
        re, im = re + [re[-1] * d[:, 0] - im[-1] * d[:, 1]], im + [re[-1] * d[:, 1] + im[-1] * d[:, 0]]
    out = [None] * (deg + 1) ** 2
    for m in range(deg + 1):
        prev2, prev = 0.0, 0.0
        for l in range(m, deg + 1):
            if l == m:
                p = torch.full_like(d[:, 0], math.prod(-(2.0 * i - 1) for i in range(1, m + 1)))
            elif l == m + 1:
                p = (2 * m + 1) * d[:, 2] * prev
            else:
                p = ((2 * l - 1) * d[:, 2] * prev - (l + m - 1) * prev2) / (l - m)
            prev2, prev = prev, p
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            if m == 0:
                out[l * l + l] = k * p
            else:
                out[l * l + l + m], out[l * l + l - m] = math.sqrt(2) * k * re[m] * p, math.sqrt(2) * k * im[m] * p
    return torch.stack(out, 1)


def _project64(s, W, cam):
    """Projected records of the Gaussians that the view sees: rows u, v, conic a, b, c,
    opacity, z, red, green, blue (differentiable), and the footprints' half extents."""
    W = torch.as_tensor(W, dtype=torch.float64, device=DEV)
    Rw, tw = W[:3, :3], W[:3, 3]
    with torch.no_grad():
        front = torch.nonzero((s["mean"] @ Rw[2] + tw[2]) > NEAR)[:, 0]
    mean, scale, quat = s["mean"][front], s["scale"][front], s["quat"][front]
    t = mean @ Rw.T + tw
    z = t[:, 2]
    q = quat / quat.norm(dim=1, keepdim=True)
    w, x, y, zz = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + zz * zz), 2 * (x * y - w * zz), 2 * (x * zz + w * y),
                       2 * (x * y + w * zz), 1 - 2 * (x * x + zz * zz), 2 * (y * zz - w * x),
                       2 * (x * zz - w * y), 2 * (y * zz + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
    M = rot * scale[:, None, :]
    lx, ly = FOV * 0.5 * cam.width / cam.fx, FOV * 0.5 * cam.height / cam.fy
    xz, yz = (t[:, 0] / z).clamp(-lx, lx), (t[:, 1] / z).clamp(-ly, ly)
    o = torch.zeros_like(z)
    J = torch.stack([cam.fx / z, o, -cam.fx * xz / z, o, cam.fy / z, -cam.fy * yz / z], 1).reshape(-1, 2, 3)
    N = J @ Rw @ M
    a, b, c = (N[:, 0] ** 2).sum(1) + EPS2D, (N[:, 0] * N[:, 1]).sum(1), (N[:, 1] ** 2).sum(1) + EPS2D
    det = a * c - b * b
    u, v = cam.fx * t[:, 0] / z + cam.cx, cam.fy * t[:, 1] / z + cam.cy
    if s["deg"] == 0:
        col = s["sh"][front][:, 0]
    else:
        d = mean + Rw.T @ tw
        d = d / d.norm(dim=1, keepdim=True)
        col = (torch.einsum("nk,nkc->nc", _sh_basis(s["deg"], d), s["sh"][front]) + 0.5).clamp(min=0)
    rec = torch.cat([torch.stack([u, v, c / det, -b / det, a / det, s["opacity"][front], z], 1), col], 1)
    with torch.no_grad():
        rx, ry = CUT * a.sqrt(), CUT * c.sqrt()
        seen = torch.nonzero((det > 0) & (u + rx >= 0) & (u - rx < cam.width) & (v + ry >= 0) & (v - ry < cam.height))[:, 0]
        near = seen[torch.sort(z[seen], stable=True).indices]
    return rec[near], rx[near], ry[near]


TILE = 16


def _tile_groups(rec, rx, ry, cam, most=24_000_000):
    """Depth-ordered lists of 16 x 16 pixel tiles, in groups of tiles with lists of like
    length: (tile numbers [B], record numbers [B][L], whether the entry is one)."""
    ntx, nty = -(-cam.width // TILE), -(-cam.height // TILE)
    u, v = rec[:, 0], rec[:, 1]
    x0, x1 = (((u + k * rx) / TILE).floor().clamp(0, ntx - 1).long() for k in (-1, 1))
    y0, y1 = (((v + k * ry) / TILE).floor().clamp(0, nty - 1).long() for k in (-1, 1))
    nx, n = x1 - x0 + 1, (x1 - x0 + 1) * (y1 - y0 + 1)
    who = torch.repeat_interleave(torch.arange(len(n), device=DEV), n)
    k = torch.arange(len(who), device=DEV) - torch.repeat_interleave(n.cumsum(0) - n, n)
    tile = (y0[who] + k // nx[who]) * ntx + x0[who] + k % nx[who]
    who = who[torch.sort(tile, stable=True).indices]
    count = torch.bincount(tile, minlength=ntx * nty)
    start = count.cumsum(0) - count
    order = torch.sort(count, descending=True, stable=True).indices
    sizes = count[order].tolist()
    i = 0
    while i < len(sizes) and sizes[i] > 0:
        take = max(1, min(len(sizes) - i, most // (sizes[i] * TILE * TILE)))
        t = order[i:i + take]
        at = torch.arange(sizes[i], device=DEV)[None, :]
        real = at < count[t][:, None]
        yield t, who[(start[t][:, None] + at).clamp(max=len(who) - 1)], real
        i += take


def _composite64(rec, group, cam, deep):
    """Front-to-back compositing of one group of tiles: [B][256][3 or 5] (RGB, depth, alpha)."""
    t, who, real = group
    ntx = -(-cam.width // TILE)
    px = torch.arange(TILE, device=DEV, dtype=torch.float64) + 0.5
    x = ((t % ntx) * TILE)[:, None] + px.repeat(TILE)[None, :]
    y = ((t // ntx) * TILE)[:, None] + px.repeat_interleave(TILE)[None, :]
    r = rec[who]
    dx, dy = x[:, None, :] - r[:, :, 0:1], y[:, None, :] - r[:, :, 1:2]
    power = -0.5 * (r[:, :, 2:3] * dx * dx + r[:, :, 4:5] * dy * dy) - r[:, :, 3:4] * dx * dy
    alpha = (r[:, :, 5:6] * torch.exp(power)).clamp(max=A_MAX)
    with torch.no_grad():
        kept = (power >= -0.5 * CUT * CUT) & (alpha >= A_MIN) & real[:, :, None]
    alpha = torch.where(kept, alpha, 0.0)
    after = torch.cumsum(torch.log1p(-alpha), 1)
    before = torch.cat([torch.zeros_like(after[:, :1]), after[:, :-1]], 1)
    w = torch.where(after.detach() >= math.log(T_MIN), alpha * torch.exp(before), 0.0).transpose(1, 2)
    what = torch.cat([r[:, :, 7:10], r[:, :, 6:7], torch.ones_like(r[:, :, :1])], 2) if deep else r[:, :, 7:10]
    return w @ what


def _render64(s, W, cam, deep=False):
    """RGB [3][H][W] of the map `s` at pose W; with `deep`, depth and alpha [H][W] too."""
    with torch.no_grad():
        rec, rx, ry = _project64(s, W, cam)
        out = _assemble(cam, 5 if deep else 3, ((g[0], _composite64(rec, g, cam, deep)) for g in _tile_groups(rec, rx, ry, cam)))
    return (out[:3], out[3], out[4]) if deep else (out[:3], None, None)


def _assemble(cam, planes, tiles):
    ntx, nty = -(-cam.width // TILE), -(-cam.height // TILE)
    out = torch.zeros((nty * ntx, TILE * TILE, planes), dtype=torch.float64, device=DEV)
    for t, c in tiles:
        out[t] = c
    out = out.reshape(nty, ntx, TILE, TILE, planes).permute(4, 0, 2, 1, 3).reshape(planes, nty * TILE, ntx * TILE)
    return out[:, :cam.height, :cam.width].contiguous()


def _cut(cam, grad, t):
    """The tiles `t` of an image gradient [planes][H][W] as _composite64 lays them out."""
    ntx, nty = -(-cam.width // TILE), -(-cam.height // TILE)
    full = torch.zeros((grad.shape[0], nty * TILE, ntx * TILE), dtype=torch.float64, device=DEV)
    full[:, :cam.height, :cam.width] = grad
    full = full.reshape(-1, nty, TILE, ntx, TILE).permute(1, 3, 2, 4, 0).reshape(nty * ntx, TILE * TILE, -1)
    return full[t]


def _backward64(s, W, cam, grad):
    """Carries an image gradient [3 or 5][H][W] of the view W back into the leaves of `s` (and W)."""
    rec, rx, ry = _project64(s, W, cam)
    leaf = rec.detach().requires_grad_()
    for g in _tile_groups(leaf.detach(), rx, ry, cam, most=6_000_000):
        out = _composite64(leaf, g, cam, grad.shape[0] == 5)
        out.backward(_cut(cam, grad, g[0]))
    rec.backward(leaf.grad)


def _ncc64(img, query):
    a, b = img.reshape(-1), query.double().reshape(-1)
    a, b = a - a.mean(), b - b.mean()
    saa, sbb = (a * a).sum(), (b * b).sum()
    if float(saa) <= 1e-12 * a.numel() or float(sbb) <= 1e-12 * a.numel():
        return 0.0 * (a * b).sum()
    return (a * b).sum() / (saa.sqrt() * sbb.sqrt())


def _grid_poses(coarse, grid):
    nx, ny, nyaw, sxy, syaw = grid
    W = _wp(coarse)
    C = -W[:3, :3].T @ W[:3, 3]
    out = []
    for k in range(nx * ny * nyaw):
        ix, iy, iw = k % nx, (k // nx) % ny, k // (nx * ny)
        psi = math.radians((iw - 0.5 * (nyaw - 1)) * syaw)
        rz = np.array([[math.cos(psi), -math.sin(psi), 0], [math.sin(psi), math.cos(psi), 0], [0, 0, 1]])
        P = np.eye(4)
        P[:3, :3] = W[:3, :3] @ rz.T
        P[:3, 3] = -P[:3, :3] @ (C + [(ix - 0.5 * (nx - 1)) * sxy, (iy - 0.5 * (ny - 1)) * sxy, 0.0])
        out.append(P)
    return np.stack(out)


def _localize64(case, query, coarse, radius, grid):
    cam = _camera(case)
    s = _subset(case, _map(case), case["store"], coarse, radius)
    poses = _grid_poses(coarse, grid)
    scores = np.array([float(_ncc64(_render64(s, p, cam)[0], query)) for p in poses])
    best = int(np.argmax(scores))
    rgb, depth, alpha = _render64(s, poses[best], cam, True)
    return {"best": best, "score": np.float64(scores[best]), "pose": poses[best], "n_gauss": int(s["mean"].shape[0]),
            "n_scored": len(poses), "scores": scores, "rgb": rgb, "depth": depth, "alpha": alpha}


def _rgb_loss(x, y):
    """0.8 mean |x - y| + 0.2 (1 - mean SSIM), the right derivative of |.| at 0; images [3][H][W]."""
    d = x - y
    l1 = torch.where(d >= 0, d, -d).mean()
    k = torch.arange(-5, 6, device=DEV, dtype=torch.float64)
    k = torch.exp(-k * k / (2 * 1.5 * 1.5))
    k = k / k.sum()

    def blur(a):
        a = torch.nn.functional.pad(a, (5, 5, 5, 5))
        a = sum(k[i] * a[:, i:i + y.shape[1], :] for i in range(11))
        return sum(k[i] * a[:, :, i:i + y.shape[2]] for i in range(11))
    mx, my = blur(x), blur(y)
    sx, sy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    ssim = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
    return 0.8 * l1 + 0.2 * (1 - ssim.mean())


def _warp64(depth, alpha, Wt, Wn, cam, It, In):
    """Image t+1 re-projected into view t by the rendered depth; image t where it has no value."""
    H, W = cam.height, cam.width
    Wt, Wn = (torch.as_tensor(m, dtype=torch.float64, device=DEV) for m in (Wt, Wn))
    at = torch.nonzero((alpha >= 0.5).detach().reshape(-1))[:, 0]
    d = depth.reshape(-1)[at] / alpha.reshape(-1)[at]
    px, py = (at % W).double(), (at // W).double()
    ray = torch.stack([(px + 0.5 - cam.cx) / cam.fx, (py + 0.5 - cam.cy) / cam.fy, torch.ones_like(px)], 1)
    P = (d[:, None] * ray - Wt[:3, 3]) @ Wt[:3, :3] @ Wn[:3, :3].T + Wn[:3, 3]
    front = torch.nonzero((P[:, 2] > NEAR).detach())[:, 0]
    at, P = at[front], P[front]
    sx, sy = cam.fx * P[:, 0] / P[:, 2] + cam.cx - 0.5, cam.fy * P[:, 1] / P[:, 2] + cam.cy - 0.5
    x0, y0 = sx.detach().floor(), sy.detach().floor()
    ok = torch.nonzero((x0 >= 0) & (x0 <= W - 2) & (y0 >= 0) & (y0 <= H - 2))[:, 0]
    at, fx, fy = at[ok], (sx - x0)[ok], (sy - y0)[ok]
    k = (y0[ok] * W + x0[ok]).long()
    I = In.reshape(3, -1)
    val = (1 - fx) * (1 - fy) * I[:, k] + fx * (1 - fy) * I[:, k + 1] + (1 - fx) * fy * I[:, k + W] + fx * fy * I[:, k + W + 1]
    return It.reshape(3, -1).index_copy(1, at, val).reshape(3, H, W)


def _train64(case, i):
    cam, n = _camera(case), case["n"]
    s = _subset(case, _map(case), "fp32", i["mid"], i["radius"])
    leaves = [s["mean"], s["scale"], s["quat"], s["opacity"], s["sh"]]
    V = case["views"]
    imgs = [torch.cat([a if a.dim() == 3 else a[None] for a in _render64(s, p, cam, True)]).requires_grad_() for p in i["poses"]]
    tg = i["targets"].double()
    loss = sum(_rgb_loss(im[:3], tg[t]) for t, im in enumerate(imgs)) / V
    for t in range(V - 1):
        warped = _warp64(imgs[t][3], imgs[t][4], i["poses"][t], i["poses"][t + 1], cam, tg[t], tg[t + 1])
        loss = loss + _rgb_loss(warped, tg[t]) / (V - 1)
    loss.backward()
    for x in leaves:
        x.requires_grad_()
    for im, p in zip(imgs, i["poses"]):
        _backward64(s, p, cam, im.grad)
    rows = torch.cat([s["mean"].grad, s["scale"].grad, s["quat"].grad, s["opacity"].grad[:, None], s["sh"].grad[:, 0]], 1).T
    # columns in the map's block order: blocks by (x, y), the map's own order inside one
    b = torch.floor(_means_on_gpu(case["map"], n, case["sh"])[:, :2].double() / BLOCK[case["map"]])
    place = torch.empty(n, dtype=torch.long, device=DEV)
    place[torch.sort(b[:, 0] * 1e6 + b[:, 1], stable=True).indices] = torch.arange(n, device=DEV)
    grad = torch.zeros((14, n), dtype=torch.float64, device=DEV)
    grad[:, place[s["index"]]] = rows
    return {"loss": np.float64(loss.item()), "grad": grad}


def _so3(phi):
    th = float(np.linalg.norm(phi))
    K = np.array([[0, -phi[2], phi[1]], [phi[2], 0, -phi[0]], [-phi[1], phi[0], 0]])
    a, b = (math.sin(th) / th, (1 - math.cos(th)) / th ** 2) if th > 1e-8 else (1 - th * th / 6, 0.5 - th * th / 24)
    return np.eye(3) + a * K + b * K @ K


def _pnp64(case, i):
    """Huber-weighted Gauss-Newton on the reprojection error of the back-projected pairs."""
    cam, W0, huber = _camera(case), i["pose"], 2.0
    d, a, pr = (i[k].cpu().numpy().astype(np.float64) for k in ("depth", "alpha", "pairs"))

    def sample(im, x, y):
        x0, y0 = np.floor(x).astype(int), np.floor(y).astype(int)
        fx, fy = x - x0, y - y0
        return ((1 - fy) * ((1 - fx) * im[y0, x0] + fx * im[y0, x0 + 1]) + fy * ((1 - fx) * im[y0 + 1, x0] + fx * im[y0 + 1, x0 + 1]))
    u, v = pr[:, 0], pr[:, 1]
    inside = (np.floor(u - 0.5) >= 0) & (np.floor(v - 0.5) >= 0) & (np.floor(u - 0.5) + 1 < cam.width) & (np.floor(v - 0.5) + 1 < cam.height)
    u, v, q = u[inside], v[inside], pr[inside, 2:]
    A = sample(a, u - 0.5, v - 0.5)
    use = A >= 0.5
    u, v, q, A = u[use], v[use], q[use], A[use]
    z = sample(d, u - 0.5, v - 0.5) / A
    X = (np.stack([z * (u - cam.cx) / cam.fx, z * (v - cam.cy) / cam.fy, z], 1) - W0[:3, 3]) @ W0[:3, :3]

    def residual(W):
        P = X @ W[:3, :3].T + W[:3, 3]
        ok = P[:, 2] > 1e-6
        P = P[ok]
        r = np.stack([cam.fx * P[:, 0] / P[:, 2] + cam.cx, cam.fy * P[:, 1] / P[:, 2] + cam.cy], 1) - q[ok]
        return P, r, np.hypot(r[:, 0], r[:, 1])

    def cost(W):
        e = residual(W)[2]
        return float(np.where(e <= huber, 0.5 * e * e, huber * (e - 0.5 * huber)).sum())
    W = np.array(W0)
    for _ in range(30):
        P, r, e = residual(W)
        wt = np.where(e <= huber, 1.0, huber / np.maximum(e, 1e-300))
        o = np.zeros(len(P))
        jp = np.stack([cam.fx / P[:, 2], o, -cam.fx * P[:, 0] / P[:, 2] ** 2, o, cam.fy / P[:, 2], -cam.fy * P[:, 1] / P[:, 2] ** 2], 1).reshape(-1, 2, 3)
        cross = np.stack([o, P[:, 2], -P[:, 1], -P[:, 2], o, P[:, 0], P[:, 1], -P[:, 0], o], 1).reshape(-1, 3, 3)
        J = np.concatenate([jp, jp @ cross], 2)
        H = np.einsum("n,nij,nik->jk", wt, J, J)
        g = np.einsum("n,nij,ni->j", wt, J, r)
        delta = np.linalg.solve(H + 1e-9 * np.trace(H) / 6 * np.eye(6), -g)
        c0, s, ok = cost(W), 1.0, False
        for _ in range(11):
            E = _so3(s * delta[3:])
            T = np.eye(4)
            T[:3, :3], T[:3, 3] = E @ W[:3, :3], E @ W[:3, 3] + s * delta[:3]
            if cost(T) < c0:
                ok = True
                break
            s *= 0.5
        if not ok:
            break
        W = T
        if np.abs(s * delta).max() < 1e-12:
            break
    e = residual(W)[2]
    return {"pose": W, "rms_px": float(np.sqrt((e * e).mean())), "cost": cost(W), "n_used": len(X)}


_PROPOSAL_SHAPES = [(32, 3, 3, 2), (32,), (64, 3, 3, 32), (64,), (64, 3, 3, 64), (64,), (128, 3, 3, 64), (128,),
                    (128, 3, 3, 128), (128,), (1024, 1536), (1024,), (64, 1024), (64,)]


def _proposal64(case, i):
    """Loss and gradients of the network at its BF16 weights, hidden activations stored in
    BF16 and the chain rule taken at the stored values."""
    flat, parts, at = torch.from_numpy(i["params"]).to(DEV), [], 0
    for shape in _PROPOSAL_SHAPES:
        n = math.prod(shape)
        p = flat[at:at + n].reshape(shape)
        parts.append((p.to(torch.bfloat16) if len(shape) > 1 else p).double().requires_grad_())
        at += n

    def store(x):
        return x + (x.detach().to(torch.float32).to(torch.bfloat16).double() - x.detach())
    x = i["x"].double().permute(0, 3, 1, 2)
    for k in range(5):
        w, b = parts[2 * k], parts[2 * k + 1]
        n, _, h, wd = x.shape
        cols = torch.nn.functional.unfold(x, 3, padding=1, stride=2)          # [n][Cin * 9][pixels]
        x = w.permute(0, 3, 1, 2).reshape(w.shape[0], -1) @ cols + b[:, None]
        x = store(torch.relu(x)).reshape(n, w.shape[0], (h + 1) // 2, (wd + 1) // 2)
    x = x.permute(0, 2, 3, 1).reshape(x.shape[0], -1)
    x = store(torch.relu(x @ parts[10].T + parts[11]))
    loss = torch.nn.functional.cross_entropy(x @ parts[12].T + parts[13], i["y"].long())
    grads = torch.autograd.grad(loss, parts)
    return {"loss": np.float64(loss.item()), "grads": torch.cat([g.reshape(-1) for g in grads])}


def exact(case, seed):
    i = _inputs(case, seed)
    path = case["path"]
    if path == "gemm":
        c = i["a"].double() @ i["b"].double().T + i["bias"].double()
        return c.clamp(min=0) if case["relu"] else c
    if path == "proposal":
        return _proposal64(case, i)
    if path == "pnp":
        return _pnp64(case, i)
    if path == "train":
        return _train64(case, i)
    if path == "search":
        return None                        # over a thousand views
    cam = _camera(case)
    if path == "render":
        s = _subset(case, _map(case), case["store"], i["at"], case["radius"])
        views = [_render64(s, p, cam, True) for p in i["poses"]]
        return {k: torch.stack([v[j] for v in views]) for j, k in enumerate(("rgb", "depth", "alpha"))}
    if path == "grad":
        s = _subset(case, _map(case), case["store"], i["at"], case["radius"])
        scores, grads = [], []
        for p in i["poses"]:
            img = _render64(s, p, cam)[0].requires_grad_()
            score = _ncc64(img, i["query"])
            score.backward()
            W = torch.as_tensor(p, dtype=torch.float64, device=DEV)
            delta = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
            o = torch.zeros((), dtype=torch.float64, device=DEV)
            K = torch.stack([o, -delta[5], delta[4], delta[5], o, -delta[3], -delta[4], delta[3], o]).reshape(3, 3)
            E = torch.eye(3, dtype=torch.float64, device=DEV) + K             # Exp to first order, exact at 0
            moved = torch.cat([E @ W[:3, :3], (E @ W[:3, 3] + delta[:3])[:, None]], 1)
            _backward64(s, moved, cam, img.grad)
            scores.append(score.item())
            grads.append(delta.grad.cpu().numpy())
        return {"scores": np.array(scores), "grads": np.stack(grads)}
    if path == "localize":
        if case["nx"] * case["ny"] * case["nyaw"] > EXACT_VIEWS:
            return None
        return _localize64(case, i["query"], i["coarse"], case["radius"], _grid(case))
    # batch, serve: the scores of all queries end to end, where every cell is rendered
    if path == "serve" or sum(q[3][0] * q[3][1] * q[3][2] for q in i["queries"]) > 3 * EXACT_VIEWS:
        return None
    each = [_localize64(case, *q) for q in i["queries"]]
    out = {k: np.stack([np.asarray(e[k]) for e in each]) for k in ("best", "score", "pose", "n_gauss", "n_scored")}
    return {**out, "scores": np.concatenate([e["scores"] for e in each]), "rgb": torch.stack([e["rgb"] for e in each]),
            "depth": torch.stack([e["depth"] for e in each])}


def _grid(case):
    return tuple(case[k] for k in ("nx", "ny", "nyaw", "step_xy", "step_yaw"))

"""Timed cases of the NeDF composition renderer: what its users have it do, through native.Renderer.

Kinds of case and what each stands for:
  query   NeDF queries on caller rays (picking, collision tests, depth look-ups of a host engine);
  frame   one composited frame (Steps 1-3) into caller device buffers;
  edit    one frame while an instance is dragged: the new transforms, then the edit frame;
  march   the plain ray-marching frame (preview without a trained NeDF, judge, speed baseline);
  grad    loss and gradient of a NeDF on caller rays and labels (a caller's own optimiser loop);
  epoch   a stretch of NeDF training: fresh labelled rays, Adam steps, the weights read back.
"""
import math
import os

import numpy as np
import torch

from paper_2308_04669_gb300 import native
from paper_2308_04669_gb300 import scenegen as sg

TRAINED = os.path.join(os.path.dirname(os.path.abspath(native.__file__)), "data", "nedf_thousand_trained.npz")
KINDS = (sg.SDF_SPHERE, sg.SDF_TORUS, sg.SDF_BOX)
PRECISION = {"fp32": native.PREC_FP32, "bf16": native.PREC_BF16, "fp8": native.PREC_FP8}
# the options of the quality frames the repository benchmarks: low-confidence answers, outliers and
# doubtful misses re-answered by the plain method, hits refined
QUALITY = dict(fallback_conf=0.9, refine_steps=4, outlier_resample=1, miss_check=64, march_steps=256, march_bisect=8)
NEDF_FLOP = 2 * (78 * 128 + 5 * 128 * 128 + 128 * 2)
NERF_FLOP = 2 * (90 * 256 + 7 * 256 * 256 + 256 * 3)
CLS_FLOP = 2 * sum(fi * fo for fi, fo in sg.cls_layers())
RADIUS = {sg.SDF_SPHERE: 0.5, sg.SDF_TORUS: 0.45, sg.SDF_BOX: 0.43}     # silhouettes, for work()

_STREAM = []


def _stream():
    """One stream for every renderer of the process, as a program that draws on one stream has."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def listed():
    return [
        # a mouse pick or a handful of collision rays: the smallest call, all latency
        {"name": "query_pick", "kind": "query", "precision": "bf16", "arch": "mlp", "hidden": 6, "width": 128, "n": 300},
        # a ragged batch of depth look-ups, about the Step-1 pairs of a 1024 x 1024 frame
        {"name": "query_bulk", "kind": "query", "precision": "bf16", "arch": "mlp", "hidden": 6, "width": 128,
         "n": 1500001},
        # the paper's classifier network, answered for a region of interest
        {"name": "query_classifier", "kind": "query", "precision": "bf16", "arch": "cls", "hidden": 0, "width": 0,
         "n": 60001},
        # a viewport thumbnail of a 48-instance scene with odd sizes
        {"name": "frame_preview", "kind": "frame", "precision": "bf16", "W": 321, "H": 181, "instances": 48,
         "lights": 2, "samples": 8, "tuned": False},
        # the repository's benchmark frame: 1024 instances, 1024 x 1024, 4 lights, schedule autotuned once
        {"name": "frame_thousand", "kind": "frame", "precision": "bf16", "W": 1024, "H": 1024, "instances": 1024,
         "lights": 4, "samples": 8, "tuned": True},
        # the large E4M3 frame: 4096 instances, 2048 x 2048, 8 lights
        {"name": "frame_large_e4m3", "kind": "frame", "precision": "fp8", "W": 2048, "H": 2048, "instances": 4096,
         "lights": 8, "samples": 8, "tuned": False},
        # a reference-precision frame (FP32 on CUDA cores)
        {"name": "frame_fp32", "kind": "frame", "precision": "fp32", "W": 256, "H": 256, "instances": 48, "lights": 2,
         "samples": 8, "tuned": False},
        # dragging one object of the benchmark scene
        {"name": "edit_drag", "kind": "edit", "precision": "bf16", "W": 1024, "H": 1024, "instances": 1024,
         "lights": 4},
        # the plain method with early termination
        {"name": "march_early_stop", "kind": "march", "precision": "bf16", "W": 512, "H": 512, "instances": 1024,
         "samples": 128, "early": True},
        # a caller's optimiser at the paper's batch size of 4096 rays
        {"name": "grad_4096", "kind": "grad", "precision": "bf16", "arch": "mlp", "hidden": 6, "width": 128, "n": 4096},
        # the same for the paper's classifier network
        {"name": "grad_classifier", "kind": "grad", "precision": "bf16", "arch": "cls", "hidden": 0, "width": 0,
         "n": 4096},
        # the repository's training schedule: batches of 65,536 rays; one pass over 2^20 fresh rays
        {"name": "train_epoch", "kind": "epoch", "precision": "bf16", "hidden": 6, "width": 128, "rays": 1 << 20,
         "batch": 65536},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "frame", "frame", "frame", "edit", "march", "grad", "grad", "epoch"])
    if kind == "query":
        if rng.random() < 0.3:
            return {"kind": kind, "precision": rng.choice(["bf16", "bf16", "fp32"]), "arch": "cls", "hidden": 0, "width": 0,
                    "n": _log(rng, 100, 60000)}
        return {"kind": kind, "precision": rng.choice(["bf16", "bf16", "fp8", "fp32"]), "arch": "mlp",
                "hidden": rng.choice([4, 6, 8]), "width": rng.choice([64, 128, 128]), "n": _log(rng, 100, 1500000)}
    if kind in ("frame", "edit", "march"):
        precision = rng.choice(["bf16", "bf16", "fp8", "fp32"] if kind == "frame" else ["bf16", "bf16", "fp8"])
        W = _log(rng, 64, {"fp32": 384, "bf16": 1400, "fp8": 1800}[precision] if kind != "march" else 640)
        H = max(48, int(W * rng.uniform(0.5, 1.0)))
        c = {"kind": kind, "precision": precision, "W": W, "H": H, "instances": _log(rng, 2, 2048)}
        if kind == "march":
            return {**c, "samples": rng.choice([48, 96, 128]), "early": True}
        c["lights"] = rng.randint(1, 6)
        return c if kind == "edit" else {**c, "samples": rng.choice([4, 7, 8, 16]), "tuned": False}
    if kind == "grad":
        if rng.random() < 0.4:
            return {"kind": kind, "precision": "bf16", "arch": "cls", "hidden": 0, "width": 0, "n": _log(rng, 200, 8192)}
        return {"kind": kind, "precision": rng.choice(["bf16", "bf16", "bf16", "fp32"]), "arch": "mlp", "hidden": rng.choice([4, 6, 8]),
                "width": rng.choice([64, 128, 128]), "n": _log(rng, 200, 65536)}
    batch = _log(rng, 1024, 65536)
    return {"kind": "epoch", "precision": "bf16", "hidden": rng.choice([4, 6]), "width": rng.choice([64, 128, 128]),
            "rays": 16 * batch, "batch": batch}


# ---- inputs -----------------------------------------------------------------------------------------
def _dims(case):
    return sg.mlp_dims(sg.NEDF_IN, case["hidden"], case["width"], 2)


def _layers(case):
    """(in, out) of the packed layers of the case's NeDF."""
    if case["arch"] == "cls":
        return [(1008, 256)] + [(256, 256)] * 32 + [(256, 65), (256, 128)]
    d = [78] + [case["width"]] * case["hidden"] + [2]
    return list(zip(d[:-1], d[1:]))


def _weights(case, seed):
    """Packed float32 weights: the trained torus network where its shape is asked for, else Xavier."""
    if case.get("arch", "mlp") == "mlp" and (case["hidden"], case["width"]) == (6, 128):
        return np.load(TRAINED)["type1"].astype(np.float32)
    g = np.random.default_rng(1000 + seed)
    cls = case.get("arch", "mlp") == "cls"
    parts = []
    for i, (fi, fo) in enumerate(_layers(case if "arch" in case else {**case, "arch": "mlp"})):
        a = math.sqrt(6.0 / (fi + fo)) * (0.5 if cls and 1 <= i <= 32 and i % 2 == 0 else 1.0)
        parts += [g.uniform(-a, a, fi * fo), g.uniform(-0.05, 0.05, fo) if cls else np.zeros(fo)]
    return np.concatenate(parts).astype(np.float32)


def _type(kind, weights, case):
    cls = case.get("arch", "mlp") == "cls"
    p = np.zeros(8, np.float32)
    p[:len(sg.DEFAULT_PARAMS[kind])] = sg.DEFAULT_PARAMS[kind]
    return sg.ObjType(kind, p, 1.0, np.full(3, 0.7, np.float32), 32 if cls else case["hidden"],
                      256 if cls else case["width"], weights, nedf_arch=sg.ARCH_CLASSIFIER if cls else sg.ARCH_REGRESSION)


def _network(case, seed):
    """A renderer that holds one type's NeDF."""
    cls = case.get("arch", "mlp") == "cls"
    r = native.Renderer(64, 64, 1, 1, case["hidden"] or 1, case["width"] or 64, precision=PRECISION[case["precision"]],
                        stream=_stream(), nedf_arch=sg.ARCH_CLASSIFIER if cls else sg.ARCH_REGRESSION)
    r.set_types([_type(sg.SDF_TORUS, _weights(case, seed), case)])
    return r


def _unit(g, n):
    v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _query_rays(n, seed):
    """Rays from outside the bound at distances of 1.5 to 40; one in twenty misses the bound clearly."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    o = _unit(g, n) * (1.5 + 38.5 * torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64) ** 2)
    u = torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64)
    miss = torch.rand(n, 1, generator=g, device="cuda") < 0.05
    # the point of the ray nearest to the centre, at right angles to the ray
    side = torch.linalg.cross(o, _unit(g, n))
    side = side / side.norm(dim=1, keepdim=True) * torch.where(miss, 1.1 + 0.35 * u, 0.97 * u.sqrt())
    dist = o.norm(dim=1, keepdim=True)
    q = side.norm(dim=1, keepdim=True)
    back = o / dist
    # o = back * dist is turned so that the ray through `side` is tangent to the sphere of radius q
    p = back * (q * q / dist) + side * torch.sqrt((1 - (q / dist) ** 2).clamp_min(0))
    d = p - o
    return o.float().contiguous(), (d / d.norm(dim=1, keepdim=True)).float().contiguous()


def _labelled_rays(n, seed):
    """Rays entering the bound sphere (cosine-weighted), labelled with the closed form of a sphere."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    o = _unit(g, n)
    d = _unit(g, n) * 0.999 - o
    o, d = o.float(), (d / d.norm(dim=1, keepdim=True)).float()
    o64, d64 = o.double(), d.double()
    d64 = d64 / d64.norm(dim=1, keepdim=True)
    b = (o64 * d64).sum(1)
    disc = 0.25 - ((o64 - b[:, None] * d64) ** 2).sum(1)
    hit = disc > 0
    m = torch.where(hit, disc.clamp_min(0).sqrt(), torch.zeros_like(b))      # t_perp - D
    return o.contiguous(), d.contiguous(), m.float().contiguous(), hit.float().contiguous()


def _scene(case, seed):
    """Seeded instances of the three trained types at the benchmark scene's density, its orbit camera
    turned about the vertical axis, ring lights."""
    n = case["instances"]
    E = 20.0 * (n / 1024.0) ** (1.0 / 3.0)
    z = np.load(TRAINED)
    types = []
    for t, k in enumerate(KINDS):
        ty = sg.make_type(k, 3, t, 6, 128, 8, 256)
        ty.nedf_w = z[f"type{t}"].astype(np.float32)
        types.append(ty)
    it, R, T, s = sg.random_instances(100 + seed, n, len(KINDS), E)
    g = np.random.default_rng(seed)
    az = g.uniform(0, 2 * math.pi)
    d = np.array([math.sqrt(2) * math.cos(az), 0.6, math.sqrt(2) * math.sin(az)])
    eye = sg.f32(3.0 * max(E, 1.2) * d / np.linalg.norm(d))
    return sg.Scene("cases", case["W"], case["H"], eye, sg.f32([0, 0, 0]), 40.0,
                    sg.ring_lights(max(E, 1.2), case.get("lights", 1)), types, it, R, T, s, half_extent=E)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "query":
        o, d = _query_rays(case["n"], seed)
        return {"kind": kind, "r": _network(case, seed), "o": o, "d": d, "out": torch.empty(case["n"], 4, device="cuda")}
    if kind == "grad":
        rays = _labelled_rays(case["n"], seed)
        w = sum(fi * fo + fo for fi, fo in _layers(case))
        return {"kind": kind, "r": _network(case, seed), "rays": rays, "grad": torch.empty(w, device="cuda")}
    if kind == "epoch":
        n = case["rays"]
        return {"kind": kind, "r": _network(case, seed), "rays": n, "batch": case["batch"], "seed": seed,
                "set": {"o": torch.empty(n, 3, device="cuda"), "d": torch.empty(n, 3, device="cuda"),
                        "m_star": torch.empty(n, device="cuda"), "hit_star": torch.empty(n, device="cuda")},
                "n": sg.mlp_param_count(_dims(case))}
    sc = _scene(case, seed)
    r = native.renderer_for(sc, precision=PRECISION[case["precision"]], stream=_stream())
    o = r.get_options()
    for k, v in QUALITY.items():
        setattr(o, k, v)
    if kind == "frame":
        o.n_shade = case["samples"]
    r.set_options(o)
    cam, lights = r.camera(sc.eye, sc.target, sc.fov_deg), r.lights(sc.lights)
    n = case["W"] * case["H"]
    s = {"kind": kind, "r": r, "cam": cam, "lights": lights, "rgba": torch.empty(n, 4, device="cuda")}
    if kind == "march":
        s["samples"], s["early"] = case["samples"], int(case["early"])
        return s
    s.update(depth=torch.empty(n, device="cuda"), id=torch.empty(n, dtype=torch.int32, device="cuda"),
             shadow=torch.empty(n, device="cuda"), out=torch.empty(n, 4, device="cuda"))
    if kind == "frame":
        if case["tuned"]:
            r.autotune(cam, lights, reps=2)
        return s
    near = int(np.argmin(((sc.inst_T - 0.5 * sc.eye) ** 2).sum(1)))          # an object in front of the camera
    r.begin_edit(cam, lights, near)
    T = sc.inst_T.copy()
    T[near] += np.float32(0.05) * np.random.default_rng(seed).uniform(-4, 4, 3).astype(np.float32)
    s["placed"] = (sc.inst_type, sc.inst_R, T, sc.inst_s)
    return s


def run(s):
    r = s["r"]
    if s["kind"] == "query":
        r.nedf_query(0, s["o"], s["d"], s["out"])
        return s["out"]
    if s["kind"] == "grad":
        return {"loss": r.loss_grad(0, *s["rays"], s["grad"]), "grad": s["grad"]}
    if s["kind"] == "epoch":
        # the end of the learning-rate decay of a training run
        r.make_labels(0, s["rays"], s["seed"], 256, 8, **s["set"])
        for _ in range(s["rays"] // s["batch"]):
            r.train_step(0, s["batch"], 1e-5)
        return {"weights": r.get_nedf_weights(0, s["n"]), **s["set"]}
    if s["kind"] == "march":
        r.render_march(s["cam"], s["samples"], s["early"], s["rgba"])
        return s["rgba"]
    if s["kind"] == "edit":
        r.set_instances(*s["placed"])
        r.render_edit(s["depth"], s["id"], s["rgba"], s["shadow"], s["out"])
    else:
        r.render(s["cam"], s["lights"], s["depth"], s["id"], s["rgba"], s["shadow"], s["out"])
    return {k: s[k] for k in ("depth", "id", "rgba", "shadow", "out")}


# ---- the work a pass cannot do without ------------------------------------------------------------------
def _counts(case):
    """(primary pairs, hit pixels, pairs whose object is met, shadow pairs) estimated with 1024 rays of one
    seeded scene: the objects as spheres of their silhouettes' size."""
    sc = _scene(case, 0)
    g = np.random.default_rng(7)
    px = g.uniform(-1, 1, (1024, 2))
    fwd = -sc.eye / np.linalg.norm(sc.eye)
    right = np.cross(fwd, [0, 1, 0])
    right /= np.linalg.norm(right)
    up = np.cross(right, fwd)
    th = math.tan(math.radians(20.0))
    d = px[:, :1] * th * case["W"] / case["H"] * right + px[:, 1:] * th * up + fwd
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    C = sc.inst_T.astype(np.float64)
    rad = np.array([RADIUS[KINDS[t]] for t in sc.inst_type])

    def near(o, d, r):
        v = C[None] - o[:, None]
        b = np.einsum("nik,nk->ni", v, d)
        p2 = (v * v).sum(2) - b * b
        return b, p2 < r * r, b - np.sqrt(np.maximum(r * r - p2, 0))
    o = np.repeat(sc.eye[None].astype(np.float64), len(d), 0)
    _, kept, _ = near(o, d, 1.0)
    _, met, t = near(o, d, rad)
    t = np.where(met, t, np.inf).min(1)
    x = (o + t[:, None] * d)[np.isfinite(t)]
    n = case["W"] * case["H"]
    shadow = 0.0
    if len(x) and case.get("lights"):
        for L in sc.lights.astype(np.float64):
            v = x - L
            ell = np.linalg.norm(v, axis=1)
            b, k, te = near(np.repeat(L[None], len(x), 0), v / ell[:, None], 1.0)
            shadow += (k & (te < ell[:, None]) & (b > -1)).sum()
    return kept.sum() * n / 1024, len(x) * n / 1024, met.sum() * n / 1024, shadow * n / 1024


def work(case):
    kind = case["kind"]
    if kind in ("query", "grad", "epoch"):
        layers = _layers(case if "arch" in case else {**case, "arch": "mlp"})
        macs, params = sum(a * b for a, b in layers), sum(a * b + b for a, b in layers)
        if kind == "query":
            return {"bytes": 40 * case["n"] + 4 * params, "flops": 2 * macs * case["n"]}
        # forward, input gradients of all layers but the first, weight gradients
        step = 2 * (3 * macs - layers[0][0] * layers[0][1])
        if kind == "grad":
            return {"bytes": 32 * case["n"] + 8 * params, "flops": step * case["n"]}
        steps = case["rays"] // case["batch"]
        return {"bytes": 32 * case["rays"] + 24 * params * steps, "flops": step * case["batch"] * steps}
    n = case["W"] * case["H"]
    pairs, hits, met, shadow = _counts(case)
    if kind == "march":
        return {"bytes": 16 * n, "flops": met * NERF_FLOP * 0.2 * case["samples"]}      # samples of some weight
    if kind == "edit":
        part = 1.0 / case["instances"]
        return {"bytes": (44 + 28) * n + 64 * case["instances"], "flops": part * (pairs * NEDF_FLOP + hits * 8 * NERF_FLOP + shadow * NEDF_FLOP)}
    return {"bytes": 44 * n + 64 * case["instances"],
            "flops": (pairs + shadow) * NEDF_FLOP + hits * case["samples"] * NERF_FLOP}


# ---- the same outputs in 64 bits (networks on given rays) ---------------------------------------------------
def _encode(x, freqs):
    f = [x]
    for fn in (torch.sin, torch.cos):
        f += [fn(x * 2.0 ** k) for k in range(freqs)]
    return torch.cat(f, 1)


def _unpack(w, layers):
    got, at = [], 0
    for fi, fo in layers:
        got.append((w[at:at + fi * fo].view(fo, fi), w[at + fi * fo:at + fi * fo + fo]))
        at += fi * fo + fo
    return got


def _chord(o, d):
    d = d / d.norm(dim=1, keepdim=True)
    b = (o * d).sum(1)
    disc = 1.0 - ((o - b[:, None] * d) ** 2).sum(1)
    sq = disc.clamp_min(0).sqrt()
    return d, (disc >= 0) & (-b + sq >= 0), (-b - sq).clamp_min(0), -b + sq, -b


def _forward(case, w, o, d):
    """The network's outputs: (m, a), or the classifier's logits (193 per ray)."""
    layers = _unpack(w, _layers(case))
    d, kept, te, tx, tp = _chord(o, d)
    if case["arch"] == "mlp":
        h = _encode(torch.cat([o + te[:, None] * d, d], 1), 6)
        for W, b in layers[:-1]:
            h = torch.relu(h @ W.T + b)
        return h @ layers[-1][0].T + layers[-1][1], kept, tp
    f = [_encode(o + (te + (tx - te) * j / 15.0)[:, None] * d, 10) for j in range(16)]
    h = torch.cat(f, 1) @ layers[0][0].T + layers[0][1]
    for k in range(16):
        (W1, b1), (W2, b2) = layers[1 + 2 * k], layers[2 + 2 * k]
        h = torch.relu(h + torch.relu(h @ W1.T + b1) @ W2.T + b2)
    return torch.cat([h @ W.T + b for W, b in layers[-2:]], 1), kept, tp


def exact(case, seed):
    """Queries and gradients; the other kinds go through a renderer's whole pipeline."""
    if case["kind"] not in ("query", "grad"):
        return None
    w = torch.from_numpy(_weights(case, seed)).cuda().double()
    if case["kind"] == "query":
        o, d = (v.double() for v in _query_rays(case["n"], seed))
        out = torch.empty(case["n"], 4, dtype=torch.float64, device="cuda")
        for i in range(0, case["n"], 1 << 15):
            y, kept, tp = _forward(case, w, o[i:i + (1 << 15)], d[i:i + (1 << 15)])
            if case["arch"] == "cls":
                c, f = y[:, 1:65].argmax(1), y[:, 65:].argmax(1)
                y = torch.stack([(128 * c + f).double() / 4096 - 1, y[:, 0]], 1)
            m, a = y[:, 0], y[:, 1]
            D = tp - m
            res = torch.stack([m, a, D, ((a > 0) & (D > 0)).double()], 1)
            none = torch.tensor([0.0, 0.0, math.inf, 0.0], dtype=torch.float64, device="cuda")
            out[i:i + (1 << 15)] = torch.where(kept[:, None], res, none)
        return out
    o, d, ms, hit = (v.double() for v in _labelled_rays(case["n"], seed))
    w.requires_grad_(True)
    total = 0.0
    bce = torch.nn.functional.binary_cross_entropy_with_logits
    for i in range(0, case["n"], 1 << 14):
        sl = slice(i, i + (1 << 14))
        y, _, _ = _forward(case, w, o[sl], d[sl])
        if case["arch"] == "mlp":
            loss = (((y[:, 0] - ms[sl]) ** 2) * hit[sl]).sum() / hit.sum()
            loss = loss + 0.1 * bce(y[:, 1], hit[sl], reduction="sum") / case["n"]
        else:
            u = (ms[sl] + 1) * 32
            c = u.floor().clamp(0, 63)
            f = ((u - c) * 128).floor().clamp(0, 127)
            one = torch.nn.functional.one_hot
            bins = bce(y[:, 1:65], one(c.long(), 64).double(), reduction="none").mean(1)
            bins = bins + bce(y[:, 65:], one(f.long(), 128).double(), reduction="none").mean(1)
            loss = (bins * hit[sl]).sum() / hit.sum() + 0.1 * bce(y[:, 0], hit[sl], reduction="sum") / case["n"]
        loss.backward()
        total += float(loss.detach())
    return {"loss": total, "grad": w.grad}

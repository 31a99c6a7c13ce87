"""The work that a user of this framework has it do, as measurable cases.

Each case is one call sequence through the public Python entry points
(``paper_2606_02226_gb300.cfs``): frames of the chaos game with their clears
and their display, batches of animation frames, stored clouds, and the learned
warm-start sampler.  Sizes are those of ``workloads.py`` (the evaluation's own
scenes), of ``bench.py`` and of the tests, or generic; ``draw`` spreads them
over the ranges that the listed cases stand for.

Work is counted as plain arithmetic: an addition, a multiplication, an
elementary function, a division and a root are one operation each; integer
work (the Philox stream, bins) is not counted.  Bytes are inputs read once and
outputs written once.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_2606_02226_gb300 import cfs
from paper_2606_02226_gb300 import workloads as W

# arithmetic of one chain op, as counted above
_OP_FLOPS = {"affine2": 8, "affine3": 18, "rotate2": 8, "rotate3": 8, "translate3": 3, "swirl": 11,
             "sinusoidal": 2, "sinusoidal3": 3, "stretch": 3, "torus": 11, "perspective": 5,
             "twist_z": 9, "bend": 7, "inversion": 16, "stars": 6, "hemisphere": 8, "bands": 3,
             "splat": 4, "reset": 0}
_H, _D_IN = 128, 64


def listed():
    return [
        # an interactive preview while a system is edited: the smallest call,
        # odd sizes, one layer cleared, rendered and shown
        {"name": "preview", "kind": "preview", "maps": 5, "points": 3001, "iters": 100,
         "burn_in": 15, "w": 321, "h": 243, "channels": 3},
        # the square primitive at its published size: a small ordinary frame
        {"name": "square", "kind": "square", "points": 1 << 16, "iters": 200, "burn_in": 20,
         "w": 512},
        # the composed 2D/3D scene, the framework's headline frame: RGBA and
        # depth layers, precise trigonometry, shown as RGBA8
        {"name": "composed", "kind": "composed", "points": 1 << 22, "iters": 500, "burn_in": 20,
         "w": 2048},
        # the many-objects scene (circle maps, stars, planet, ring) at full HD
        {"name": "space", "kind": "space", "points": 1 << 20, "iters": 200, "burn_in": 20,
         "w": 1920, "h": 1080, "stars": 400},
        # an animation of 256 uneven frames in one batch, each shown as RGBA8:
        # the largest job
        {"name": "animation", "kind": "animation", "frames": 256, "lo": 16, "hi": 22,
         "iters": 300, "burn_in": 20, "res_lo": 256, "res_hi": 2048},
        # a live set of small frames from a host that may not allocate
        {"name": "realtime", "kind": "realtime", "frames": 24, "lo": 12, "hi": 17, "iters": 150,
         "burn_in": 18, "res_lo": 128, "res_hi": 512},
        # making the stored cloud of the staged alternative
        {"name": "cloud_make", "kind": "cloud_make", "points": 1 << 26, "iters": 32, "maps": 8},
        # one deformed frame of the stored cloud into a large depth layer
        {"name": "cloud_frame", "kind": "cloud_frame", "points": 1 << 26, "w": 8192, "frame": 21,
         "fold": True, "fast_trig": False},
        # putting a stored cloud into Morton order
        {"name": "cloud_order", "kind": "cloud_order", "points": (1 << 24) + 1237, "dim": 3},
        # warm-start points for every frame of an animation
        {"name": "warm_start", "kind": "warm_start", "frames": 256, "samples": 4096,
         "even": True},
        # forward, loss and backward of the sampler's training batch
        {"name": "sampler_grad", "kind": "sampler_grad", "systems": 64, "points": 1024,
         "proj": 64},
        # a stretch of training steps through the training call
        {"name": "sampler_train", "kind": "sampler_train", "systems": 64, "points": 1024,
         "proj": 64, "steps": 40, "family": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice([c["kind"] for c in listed()])
    if kind == "preview":
        return {"kind": kind, "maps": rng.randint(2, 8), "points": _log(rng, 500, 60000),
                "iters": rng.randint(40, 160), "burn_in": rng.randint(8, 24),
                "w": rng.randint(100, 800), "h": rng.randint(100, 600),
                "channels": rng.randint(1, 4)}
    if kind == "square":
        return {"kind": kind, "points": _log(rng, 1 << 14, 1 << 21),
                "iters": 4 * rng.randint(25, 75) + rng.choice([0, 0, 1]),
                "burn_in": rng.choice([16, 20, 21, 24]), "w": rng.choice([256, 512, 700, 1024])}
    if kind == "composed":
        return {"kind": kind, "points": _log(rng, 1 << 16, 1 << 21),
                "iters": rng.choice([200, 300, 402, 500]), "burn_in": 20,
                "w": rng.choice([512, 1000, 1024, 2048])}
    if kind == "space":
        w, h = rng.choice([(640, 360), (1280, 720), (1366, 768), (1920, 1080)])
        return {"kind": kind, "points": _log(rng, 1 << 15, 1 << 20), "iters": rng.choice([150, 200]),
                "burn_in": 20, "w": w, "h": h, "stars": rng.choice([60, 400, 900])}
    if kind == "animation":
        lo = rng.randint(13, 17)
        return {"kind": kind, "frames": _log(rng, 3, 96), "lo": lo, "hi": rng.randint(lo + 1, 21),
                "iters": rng.choice([150, 200, 300, 301]), "burn_in": rng.choice([18, 20]),
                "res_lo": 256, "res_hi": rng.choice([512, 1024, 2048])}
    if kind == "realtime":
        lo = rng.randint(10, 14)
        return {"kind": kind, "frames": _log(rng, 1, 128), "lo": lo, "hi": rng.randint(lo + 1, 19),
                "iters": rng.randint(80, 250), "burn_in": rng.randint(12, 24), "res_lo": 128,
                "res_hi": rng.choice([256, 512, 1024])}
    if kind == "cloud_make":
        return {"kind": kind, "points": _log(rng, 1 << 14, 1 << 25), "iters": rng.randint(20, 50),
                "maps": 8}
    if kind == "cloud_frame":
        return {"kind": kind, "points": 4 * _log(rng, 1 << 14, 1 << 23),
                "w": rng.choice([1024, 2048, 4096, 8192]), "frame": rng.randint(0, 63),
                "fold": rng.random() < 0.7, "fast_trig": rng.random() < 0.25}
    if kind == "cloud_order":
        return {"kind": kind, "points": _log(rng, 1 << 12, 1 << 25), "dim": rng.choice([2, 3])}
    if kind == "warm_start":
        return {"kind": kind, "frames": _log(rng, 1, 256), "samples": _log(rng, 100, 8000),
                "even": rng.random() < 0.3}
    if kind == "sampler_grad":
        return {"kind": kind, "systems": _log(rng, 2, 64), "points": rng.choice([64, 256, 512, 1024]),
                "proj": rng.choice([16, 33, 64])}
    return {"kind": "sampler_train", "systems": rng.choice([16, 33, 64]),
            "points": rng.choice([256, 512, 1024]), "proj": rng.choice([32, 64]),
            "steps": rng.randint(10, 40), "family": rng.randint(50, 512)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _affine_system(maps: int, seed: int) -> W.System:
    """Contractive affine maps drawn as the animation's keyframes are."""
    rng = np.random.default_rng([seed, 7101])
    ms, probs = [], []
    for _ in range(maps):
        th, s, b = rng.uniform(0, 2 * math.pi), rng.uniform(0.3, 0.7, 2), rng.uniform(-1, 1, 2)
        c, n = math.cos(th), math.sin(th)
        ms.append(W.Map("affine", tuple(W.f32(v) for v in (c * s[0], -n * s[1], n * s[0], c * s[1],
                                                            b[0], b[1]))))
        probs.append(max(s[0] * s[1], 1e-6))
    return W.System(2, ms, probs)


def _frames(case, seed):
    """Uneven frames of an animation: their sizes belong to the case, their
    systems to the seed."""
    res = [r for r in (128, 256, 512, 1024, 2048) if case["res_lo"] <= r <= case["res_hi"]]
    sizes = W.animation_frames(case["frames"], seed=0, min_log2=case["lo"], max_log2=case["hi"],
                               resolutions=tuple(res))
    systems = W.animation_frames(case["frames"], seed=seed)
    return [replace(a, system=b.system, t=b.t) for a, b in zip(sizes, systems)]


def _slices(shapes, dtype, fill=None):
    """Tensors of the given shapes in one allocation, each 256-byte aligned."""
    sizes = [-(-int(np.prod(s)) // 64) * 64 for s in shapes]
    flat = torch.zeros(sum(sizes), dtype=dtype, device="cuda")
    out, at = [], 0
    for s, n in zip(shapes, sizes):
        out.append(flat[at:at + int(np.prod(s))].view(s))
        at += n
    return flat, out


def _weights(seed):
    """A network's parameters at the scale of its initialisation, with biases."""
    rng = np.random.default_rng([seed, 7102])
    parts = []
    for o, i in ((_H, _D_IN), (_H, _H), (_H, _H), (2, _H)):
        b = 1.0 / math.sqrt(i)
        parts += [rng.uniform(-b, b, o * i), rng.uniform(-b, b, o) * 0.5]
    return np.concatenate(parts).astype(np.float32)


def _target(w, h, channels, view):
    return W.Target("hist_u32", w, h, channels, view, palette=W.palette_rgba(W.MAX_MAPS))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed, "kind": kind}
    if kind in ("preview", "square", "composed", "space"):
        if kind == "preview":
            jobs = [W.RenderJob(_affine_system(case["maps"], seed), 0, case["points"])]
            chain = [W.Op("splat", (0,))]
            descs = [_target(case["w"], case["h"], case["channels"], W.ANIMATION_VIEW)]
        elif kind == "square":
            wl = W.square_render(case["points"], case["iters"], case["burn_in"], case["w"])
            jobs, chain, descs = wl.jobs, wl.chain, wl.targets
        elif kind == "composed":
            wl = W.composed_render(case["points"], case["iters"], case["burn_in"], case["w"])
            jobs, chain, descs = wl.jobs, wl.chain, wl.targets
        else:
            wl = W.space_render(case["points"], case["iters"], case["burn_in"], case["w"],
                                case["h"], n_stars=case["stars"])
            jobs, chain, descs = wl.jobs, wl.chain, wl.targets
        s["descs"] = descs
        s["chain"] = cfs.Chain(chain, 2, fold_linear=kind == "space")
        s["jobs"] = [(cfs.System(j.system), j.point_begin, j.n_points) for j in jobs]
        s["tens"] = [cfs.alloc_target(d) for d in descs]
        s["disc"] = torch.zeros(len(descs), dtype=torch.int64, device="cuda")
        s["rgba8"] = torch.zeros((descs[0].H, descs[0].W), dtype=torch.int32, device="cuda")
        s["a_max"] = torch.zeros(1, dtype=torch.float32, device="cuda")
        for sy, _, _ in s["jobs"]:
            cfs.prepare(sy, s["chain"], descs, s["tens"])
    elif kind in ("animation", "realtime"):
        fr = _frames(case, seed)
        descs = [replace(W.animation_target(f.W), palette=W.palette_rgba(W.MAX_MAPS)) for f in fr]
        s["hist"], hists = _slices([(4, f.W, f.W) for f in fr], torch.int32)
        s["frames"] = [(cfs.System(f.system), f.n_points, 0, j, [d], [h])
                       for j, (f, d, h) in enumerate(zip(fr, descs, hists))]
        s["disc"] = torch.zeros(len(fr), dtype=torch.int64, device="cuda")
        if kind == "animation":
            s["batch"] = cfs.Batch(cfs.Chain([W.Op("splat", (0,))], 2), s["frames"],
                                   iters=case["iters"], burn_in=case["burn_in"], seed=seed)
            s["rgba8"], s["outs"] = _slices([(f.W, f.W) for f in fr], torch.int32)
    elif kind == "cloud_make":
        s["system"] = cfs.System(W.cloud_system(seed))
        s["xyz"] = torch.zeros((3, case["points"]), dtype=torch.float32, device="cuda")
        s["fn"] = torch.zeros(case["points"], dtype=torch.uint8, device="cuda")
    elif kind == "cloud_frame":
        s["xyz"], s["fn"] = cfs.pointcloud_generate(cfs.System(W.cloud_system(seed)),
                                                    case["points"], 32, seed=seed)
        s["chain"] = cfs.Chain(W.cloud_chain(case["frame"], seed=seed), 3,
                               fast_trig=case["fast_trig"], fold_linear=case["fold"])
        s["descs"] = [W.cloud_target(case["w"])]
        s["tens"] = [cfs.alloc_target(s["descs"][0])]
        s["disc"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    elif kind == "cloud_order":
        sy = W.cloud_system(seed) if case["dim"] == 3 else _affine_system(6, seed)
        s["xyz"], s["fn"] = cfs.pointcloud_generate(cfs.System(sy), case["points"], 32, seed=seed)
    elif kind == "warm_start":
        fr = W.animation_frames(case["frames"], seed=seed)
        rng = np.random.default_rng([case["frames"], 7103])     # sizes belong to the case
        ms = [case["samples"] if case["even"] else max(1, int(case["samples"] * rng.uniform(0.5, 1)))
              for _ in fr]
        s["sampler"] = cfs.Sampler(_weights(seed))
        s["systems"], s["descr"] = [cfs.System(f.system) for f in fr], [f.system for f in fr]
        s["t"], s["seeds"], s["ms"] = [f.t for f in fr], [seed * 1000 + j for j in range(len(fr))], ms
        s["flat"], s["outs"] = _slices([(2, m) for m in ms], torch.float32)
    elif kind == "sampler_grad":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        S, N = case["systems"], case["points"]
        s["params"] = _weights(seed)
        s["sampler"] = cfs.Sampler(s["params"])
        U = torch.zeros((S, N, _D_IN), device="cuda")
        U[..., 0:2] = torch.randn((S, N, 2), generator=g, device="cuda")
        U[..., 2:51] = (2 * torch.rand((S, 1, 49), generator=g, device="cuda") - 1)
        s["U"] = U.reshape(S * N, _D_IN).to(torch.bfloat16)
        s["T"] = torch.randn((S, N, 2), generator=g, device="cuda") * 0.8 + 0.3
        s["phi"] = ((torch.arange(case["proj"], device="cuda") + 0.37) *
                    (2 * math.pi / case["proj"])).float()
    else:                                                   # sampler_train
        fr = W.animation_frames(case["family"], seed=seed + 1)
        s["params"] = _weights(seed)
        s["sampler"] = cfs.Sampler(s["params"])
        s["zeros"] = np.zeros_like(s["params"])
        s["systems"], s["t"] = [cfs.System(f.system) for f in fr], [f.t for f in fr]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c, kind = s["case"], s["kind"]
    if kind in ("preview", "square", "composed", "space"):
        cfs.target_clear(s["descs"], s["tens"])
        s["disc"].zero_()
        for j, (sy, begin, n) in enumerate(s["jobs"]):
            cfs.render(sy, s["chain"], s["descs"], s["tens"], n_points=n, point_begin=begin,
                       iters=c["iters"], burn_in=c["burn_in"], seed=s["seed"], system_id=j,
                       discards=s["disc"])
        if kind == "square":
            return [s["tens"][0], s["disc"]]
        cfs.tonemap(s["descs"][0], s["tens"][0], s["rgba8"], a_max_out=s["a_max"])
        return [*s["tens"], s["disc"], s["rgba8"]]
    if kind == "animation":
        s["batch"].launch(clear=True)
        s["batch"].display(s["outs"])
        return [s["hist"], s["rgba8"]]
    if kind == "realtime":
        cfs.render_batch_noalloc(s["frames"], iters=c["iters"], burn_in=c["burn_in"],
                                 seed=s["seed"], discards=s["disc"])
        return [s["hist"], s["disc"]]
    if kind == "cloud_make":
        cfs.pointcloud_generate(s["system"], c["points"], c["iters"], seed=s["seed"], xyz=s["xyz"],
                                fn=s["fn"])
        return [s["xyz"], s["fn"]]
    if kind == "cloud_frame":
        cfs.target_clear(s["descs"], s["tens"])
        s["disc"].zero_()
        cfs.render_points(s["chain"], s["xyz"], s["fn"], s["descs"], s["tens"], discards=s["disc"])
        return [s["tens"][0], s["disc"]]
    if kind == "cloud_order":
        return list(cfs.pointcloud_reorder(s["xyz"], s["fn"]))
    if kind == "warm_start":
        s["sampler"].start_points_batch(s["systems"], s["t"], s["outs"], s["seeds"])
        return [s["flat"]]
    if kind == "sampler_grad":
        Y = s["sampler"].forward(s["U"])
        loss, dX = cfs.sw_loss(Y.view(c["systems"], c["points"], 2), s["T"], s["phi"])
        grads = s["sampler"].backward(s["U"], dX)
        return [Y, loss, dX, grads]
    s["sampler"].set_params(s["params"], s["zeros"], s["zeros"], 0)
    hist = s["sampler"].train(s["systems"], s["t"], c["steps"], systems_per_step=c["systems"],
                              points_per_system=c["points"], n_proj=c["proj"], seed=s["seed"])
    return [hist, s["sampler"].get_params()[0]]


# ---------------------------------------------------------------------------
# work a pass cannot do without
# ---------------------------------------------------------------------------
def _layer_bytes(d):
    return d.W * d.H * {"hist_u32": 4 * d.C, "rgba_f32": 16, "depth_u64": 8}[d.kind]


def work(case):
    kind = case["kind"]
    steps = case.get("iters", 0)
    splats = max(0, steps - case.get("burn_in", 0))
    if kind in ("preview", "square", "composed", "space"):
        gen = 13 if kind == "space" else 8
        chain = {"preview": [W.Op("splat")], "square": [W.Op("splat")],
                 "composed": W.composed_chain(), "space": W.space_chain()}[kind]
        descs = {"preview": lambda: [_target(case["w"], case["h"], case["channels"], (0, 1, 0, 1))],
                 "square": lambda: [W.Target("hist_u32", case["w"], case["w"], 4)],
                 "composed": lambda: W.composed_targets(case["w"]),
                 "space": lambda: [W.space_target(case["w"], case["h"])]}[kind]()
        px = descs[0].W * descs[0].H
        return {"bytes": sum(map(_layer_bytes, descs)) + (0 if kind == "square" else 4 * px),
                "flops": case["points"] * (steps * gen + splats * sum(_OP_FLOPS[o.kind]
                                                                      for o in chain))}
    if kind in ("animation", "realtime"):
        fr = _frames(case, 1)
        px, n = sum(f.W * f.W for f in fr), sum(f.n_points for f in fr)
        return {"bytes": px * (20 if kind == "animation" else 16),
                "flops": n * (8 * steps + 4 * splats)}
    n = case.get("points", 0)
    if kind == "cloud_make":
        return {"bytes": 13 * n, "flops": 18 * n * steps}
    if kind == "cloud_frame":
        ops = sum(_OP_FLOPS[o.kind] for o in W.cloud_chain(case["frame"]))
        return {"bytes": 13 * n + 8 * case["w"] ** 2, "flops": n * ops}
    if kind == "cloud_order":
        return {"bytes": 2 * (4 * case["dim"] + 1) * n, "flops": 0}
    weights = _H * _D_IN + 2 * _H * _H + 2 * _H
    if kind == "warm_start":
        rows = case["frames"] * case["samples"]
        return {"bytes": 8 * rows, "flops": 2 * rows * (2 * _H + 2 * _H * _H + 2 * _H)}
    rows = case["systems"] * n
    net, sort = 6 * rows * weights, rows * case["proj"] * (2 * math.log2(n) + 12)
    if kind == "sampler_grad":
        return {"bytes": rows * (2 * _D_IN + 8 + 8 + 8) + 8 * weights, "flops": net + sort}
    return {"bytes": 16 * weights, "flops": case["steps"] * (net + sort + rows * 40 * 8)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the documented rules alone
# ---------------------------------------------------------------------------
def _philox(c, seed):
    """Philox4x32-10 of the four counter words ``c`` (int64 tensors holding
    u32 values) with the key (seed low, seed high)."""
    M = 0xFFFFFFFF
    k0, k1 = seed & M, (seed >> 32) & M
    c0, c1, c2, c3 = c
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & M) ^ c1 ^ k0, p1 & M, ((p0 >> 32) & M) ^ c3 ^ k1, p0 & M)
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _exact_cloud(case, seed):
    d = W.cloud_system(seed)
    n, m = case["points"], len(d.maps)
    run_sum, total, th = 0.0, sum(d.probs), []
    for p in d.probs[:-1]:
        run_sum += p
        th.append(math.floor(run_sum / total * 2.0 ** 32))
    prm = torch.tensor([mp.params for mp in d.maps], dtype=torch.float64, device="cuda")
    T = torch.tensor(th, dtype=torch.int64, device="cuda")
    out = torch.empty((3, n), dtype=torch.float64, device="cuda")
    for a in range(0, n, 1 << 22):
        i = torch.arange(a, min(n, a + (1 << 22)), dtype=torch.int64, device="cuda")
        z = torch.zeros_like(i)
        w = _philox((i, z, z, z + 1), seed)
        p = [(w[d_] >> 8).double() * 2.0 ** -24 for d_ in range(3)]
        for step in range(case["iters"]):
            if step % 4 == 0:
                w = _philox((i, z + step // 4, z, z), seed)
            q = prm[torch.bucketize(w[step % 4], T, right=True).clamp_(max=m - 1)]
            p = [q[:, 3 * r] * p[0] + q[:, 3 * r + 1] * p[1] + q[:, 3 * r + 2] * p[2] + q[:, 9 + r]
                 for r in range(3)]
        for r in range(3):
            out[r, a:a + i.numel()] = p[r]
    return [out, None]


def _exact_order(case, seed):
    s = prepare(case, seed)
    x, dim = s["xyz"], case["dim"]
    key = torch.zeros(x.shape[1], dtype=torch.int64, device="cuda")
    for d in range(dim):
        lo, hi = x[d].min(), x[d].max()
        q = ((x[d] - lo) * (torch.tensor(1024.0, device="cuda") / (hi - lo))).to(torch.int64)
        q = q.clamp_(0, 1023)
        for b in range(10):
            key |= ((q >> b) & 1) << (dim * b + d)
    perm = torch.argsort(key, stable=True)
    return [x[:, perm].double(), None]


def _layers(params):
    at, out = 0, []
    for o, i in ((_H, _D_IN), (_H, _H), (_H, _H), (2, _H)):
        w = torch.tensor(params[at:at + o * i], dtype=torch.float64, device="cuda").view(o, i)
        b = torch.tensor(params[at + o * i:at + o * i + o], dtype=torch.float64, device="cuda")
        out.append((w, b))
        at += o * i + o
    return out


def _forward(layers, u):
    for j, (w, b) in enumerate(layers):
        u = u @ w.T + b
        if j < 3:
            u = u * torch.sigmoid(u)
    return u


def _exact_warm(case, seed):
    s = prepare(case, seed)
    layers = _layers(_weights(seed))
    flat, outs = _slices([(2, m) for m in s["ms"]], torch.float64)
    for d, t, m, sd, out in zip(s["descr"], s["t"], s["ms"], s["seeds"], outs):
        maps = [np.asarray(q.params, np.float64) for q in d.maps]
        order = sorted(range(len(maps)), key=lambda k: (-abs(maps[k][0] * maps[k][3] -
                                                             maps[k][1] * maps[k][2]), k))
        cond = np.zeros(_D_IN - 2)
        for q, k in enumerate(order):
            cond[6 * q:6 * q + 6] = maps[k][:6]
        cond[48] = t
        i = torch.arange(m, dtype=torch.int64, device="cuda")
        z = torch.zeros_like(i)
        w = _philox((i, z, z, z + 3), sd)
        u1, u2 = ((w[0] >> 8).double() + 0.5) * 2.0 ** -24, (w[1] >> 8).double() * 2.0 ** -24
        r = torch.sqrt(-2 * torch.log(u1))
        u = torch.zeros((m, _D_IN), dtype=torch.float64, device="cuda")
        u[:, 0], u[:, 1] = r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)
        u[:, 2:] = torch.tensor(cond, device="cuda")
        out.copy_(_forward(layers, u).T)
    return [flat]


def _exact_grad(case, seed):
    s = prepare(case, seed)
    S, N, P = case["systems"], case["points"], case["proj"]
    leaves = [(w.requires_grad_(), b.requires_grad_()) for w, b in _layers(s["params"])]
    Y = _forward(leaves, s["U"].double())
    X = Y.detach().view(S, N, 2)
    th = torch.stack([torch.cos(s["phi"].double()), torch.sin(s["phi"].double())])
    px, order = (X @ th).sort(dim=1)
    diff = px - (s["T"].double() @ th).sort(dim=1).values
    loss = (diff * diff).mean(dim=1).mean()
    g = torch.zeros_like(diff).scatter_(1, order, 2 * diff / N) / (S * P)
    dX = g @ th.T
    Y.backward(dX.view(S * N, 2))
    grads = torch.cat([v.grad.reshape(-1) for wb in leaves for v in wb])
    return [Y.detach(), loss.view(1), dX, grads]


def exact(case, seed):
    """Outputs in 64 bits for the paths whose results are computed numbers and
    do not hang on single rounding decisions (a histogram's bins do: those
    layers are whole numbers, and sums of them)."""
    f = {"cloud_make": _exact_cloud, "cloud_order": _exact_order, "warm_start": _exact_warm,
         "sampler_grad": _exact_grad}.get(case["kind"])
    return f(case, seed) if f else None

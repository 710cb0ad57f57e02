"""What the library is timed on: its public calls, over the sizes and options they are used with.

A case is a dict of plain values; ``kind`` names the call:

  static    cvo_eval_gradient_static: the allocation-free gradient pass on device tensors
  eval      Context.eval: F, gradient and step sums of two resident clouds at one pose
  align     Context.align: a whole solve of two resident clouds from the identity
  track     the per-frame step of a tracker: upload a frame from host arrays, align it to the
            resident keyframe, release it
  batch     Batch.run: many uneven pairs in one launch
  serve     the request loop: a burst of frames of several cameras submitted and polled to the end
  frontend  Context.frontend_select: the points of one RGB-D frame

Clouds are synthetic: three textured planes of 2 m ("planes"), or frames ray-cast in a textured
room of 6 x 5 x 3 m and cut to the pixels of high intensity gradient ("room").

The pair sums, and so F, gradients, step sums and the poses that follow from them, are formed in
FP32 and handed back in C doubles; ``run`` returns them in the type in which they are formed.
"""
import math
import random
import time

import numpy as np
import torch

import paper_1904_02266_gb300 as cvo

DEV = "cuda"
KERNEL, DOT, NONE = "kernel", "dot", "none"
MODES = {KERNEL: cvo.CVO_COLOR_KERNEL, DOT: cvo.CVO_COLOR_DOT, NONE: cvo.CVO_COLOR_NONE}


def listed():
    return [
        # a real-time loop that may not allocate scores one pose of a few hundred points: the
        # smallest call, bound by launches
        {"name": "static_600", "kind": "static", "n": 500, "m": 600, "dim": 5, "mode": KERNEL, "ell": 0.1},
        # the same entry point on whole semi-dense frames
        {"name": "static_20k", "kind": "static", "n": 20000, "m": 20000, "dim": 5, "mode": KERNEL, "ell": 0.06},
        # one pose scored on small resident clouds (relocalisation asks this many times)
        {"name": "eval_2k", "kind": "eval", "scene": "planes", "n": 2000, "m": 2000, "dim": 5, "mode": KERNEL,
         "bf16": 0, "ell": 0.15},
        # odd sizes, eight features and the paper's dot-product labels
        {"name": "eval_20k_dot8", "kind": "eval", "scene": "room", "n": 20011, "m": 17333, "dim": 8, "mode": DOT,
         "bf16": 0, "ell": 0.06},
        # dense frames with features stored in BF16
        {"name": "eval_100k_bf16", "kind": "eval", "scene": "room", "n": 100000, "m": 100000, "dim": 5,
         "mode": KERNEL, "bf16": 1, "ell": 0.05},
        # small pair: 2000 points on three planes
        {"name": "align_2k", "kind": "align", "scene": "planes", "n": 2000, "m": 2000, "dim": 5, "mode": KERNEL,
         "bf16": 0},
        # the benchmark's pair: semi-dense VGA frames of 20k points
        {"name": "align_room_20k", "kind": "align", "scene": "room", "n": 20000, "m": 20000, "dim": 5,
         "mode": KERNEL, "bf16": 0},
        # dense VGA frames
        {"name": "align_room_100k", "kind": "align", "scene": "room", "n": 100000, "m": 100000, "dim": 5,
         "mode": KERNEL, "bf16": 0},
        # a camera frame against its keyframe, from host memory, as a tracker runs it
        {"name": "track_20k", "kind": "track", "scene": "room", "n": 20000, "m": 19001, "dim": 5, "mode": KERNEL,
         "bf16": 0},
        # offline registration: uneven pairs in one launch, each with its own first lengthscale
        {"name": "batch_64", "kind": "batch", "pairs": 64, "lo": 2000, "hi": 40000, "dim": 5, "mode": KERNEL,
         "bf16": 0},
        # continuous batching: a burst of frames of four cameras
        {"name": "serve_16", "kind": "serve", "requests": 16, "cameras": 4, "lo": 5000, "hi": 60000, "dim": 5,
         "mode": KERNEL, "bf16": 0},
        # semi-dense points of one VGA frame
        {"name": "frontend_vga", "kind": "frontend", "width": 640, "height": 480, "percentile": 80.0,
         "max_points": 0},
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n | 1 if rng.random() < 0.5 else n

    def ell(lo, hi):
        return round(math.exp(rng.uniform(math.log(lo), math.log(hi))), 4)

    kind = rng.choice(("static", "static", "eval", "eval", "eval", "align", "align", "track", "batch", "serve",
                       "frontend"))
    if kind == "frontend":
        w = rng.randint(160, 1024)
        return {"kind": kind, "width": w, "height": w * 3 // 4 - rng.randint(0, 7),
                "percentile": round(rng.uniform(50.0, 95.0), 1), "max_points": rng.choice((0, 5000, 20000))}
    dim, mode = rng.choice(((5, KERNEL), (5, KERNEL), (5, KERNEL), (3, KERNEL), (8, KERNEL), (0, NONE)))
    if kind in ("static", "eval") and dim and rng.random() < 0.25:
        mode = DOT
    if kind == "static":
        n = size(300, 20000)
        m = max(300, min(20000, int(n * rng.uniform(0.7, 1.4))))
        return {"kind": kind, "n": n, "m": m, "dim": dim, "mode": mode, "ell": ell(0.03, 0.15)}
    bf16 = 1 if dim and rng.random() < 0.25 else 0
    if kind == "batch":
        lo = size(1000, 5000)
        return {"kind": kind, "pairs": rng.randint(5, 48), "lo": lo, "hi": lo + size(1000, 35000), "dim": dim,
                "mode": mode, "bf16": bf16}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(4, 16), "cameras": rng.randint(1, 4), "lo": size(2000, 6000),
                "hi": size(10000, 60000), "dim": dim, "mode": mode, "bf16": bf16}
    n = size(1000, 60000)
    c = {"kind": kind, "scene": "planes" if n < 4000 or rng.random() < 0.4 else "room", "n": n,
         "m": max(1000, min(60000, int(n * rng.uniform(0.7, 1.3)))), "dim": dim, "mode": mode, "bf16": bf16}
    if kind == "eval":
        c["ell"] = ell(0.02, 0.15)
    return c


# ---- scenes ----------------------------------------------------------------------------------

def _rigid(rng, deg, metres):
    """A rotation of deg degrees about a random axis and a translation of the given length."""
    a, t = rng.normal(size=3), rng.normal(size=3)
    a, t = a / np.linalg.norm(a), t * (metres / np.linalg.norm(t))
    th = math.radians(deg)
    W = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    P = np.eye(4)
    P[:3, :3] = np.eye(3) + math.sin(th) * W + (1 - math.cos(th)) * (W @ W)
    P[:3, 3] = t
    return P


def _move(P, x):
    M = torch.as_tensor(P, device=DEV, dtype=torch.float64)
    return x @ M[:3, :3].T + M[:3, 3]


def _textures(rng, faces):
    """Three sinusoids per face: wave vectors of 1 to 4 cycles a metre and phases."""
    ang, mag = rng.uniform(0, 2 * np.pi, (faces, 3)), rng.uniform(1.0, 4.0, (faces, 3))
    k = np.stack([mag * np.cos(ang), mag * np.sin(ang)], axis=-1)
    return [torch.as_tensor(v, device=DEV) for v in (k, rng.uniform(0, 2 * np.pi, (faces, 3)))]


def _planes(tex, n, gen):
    """n noisy points on three orthogonal planes, with H, S, V and the slope of V as features."""
    k, phi = tex
    face = torch.arange(n, device=DEV) % 3
    uv = 2.0 * torch.rand(n, 2, generator=gen, device=DEV, dtype=torch.float64)
    pts = torch.zeros(n, 3, device=DEV, dtype=torch.float64)
    for f, (a, b) in enumerate(((1, 2), (0, 2), (0, 1))):
        on = face == f
        pts[on, a], pts[on, b] = uv[on, 0], uv[on, 1]
    pts += 0.005 * torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)
    kf = k[face]
    phase = 2 * np.pi * (kf * uv[:, None, :]).sum(-1) + phi[face]
    kv = kf[:, 2, :]
    slope = torch.cos(phase[:, 2])[:, None] * kv / kv.norm(dim=1, keepdim=True)
    return pts, torch.cat([0.5 + 0.5 * torch.sin(phase), slope], dim=1)


class _Room:
    """A 6 x 5 x 3 m room with 20 boxes, each face textured."""

    def __init__(self, rng):
        self.cam = np.array([rng.uniform(0.6, 1.0), rng.uniform(2.0, 3.0), rng.uniform(1.2, 1.6)])
        lo, hi = [np.zeros(3)], [np.array([6.0, 5.0, 3.0])]
        while len(lo) < 21:
            dims = rng.uniform(0.2, (1.0, 1.0, 1.5))
            pos = np.append(rng.uniform(0.0, hi[0][:2] - dims[:2]), 0.0)
            if np.linalg.norm(np.clip(self.cam, pos, pos + dims) - self.cam) >= 1.0:
                lo.append(pos)
                hi.append(pos + dims)
        self.lo, self.hi = (torch.as_tensor(np.array(v), device=DEV) for v in (lo, hi))
        self.tex = _textures(rng, 6 * len(lo))
        yaw, pitch = rng.uniform(-0.35, 0.35), rng.uniform(-0.25, -0.05)
        cy, sy, cp, sp = math.cos(yaw), math.sin(yaw), math.cos(pitch), math.sin(pitch)
        self.T = np.eye(4)
        self.T[:3, :3] = (np.array([[cy, -sy, 0], [sy, cy, 0], [0, 0, 1.0]]) @
                          np.array([[cp, 0, sp], [0, 1.0, 0], [-sp, 0, cp]]) @
                          np.array([[0, 0, 1.0], [-1.0, 0, 0], [0, -1.0, 0]]))
        self.T[:3, 3] = self.cam

    def render(self, T, W, H, gen):
        """Depth with 1% noise (0 outside 0.5 to 5 m), HSV colour and the rays of one frame."""
        f = 525.0 * W / 640.0
        v, u = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64),
                              torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
        ray = torch.stack([(u - (W - 1) / 2) / f, (v - (H - 1) / 2) / f, torch.ones_like(u)], -1).reshape(-1, 3)
        T = torch.as_tensor(T, device=DEV)
        d, o = ray @ T[:3, :3].T, T[:3, 3]
        d = torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
        best = torch.full((d.shape[0],), math.inf, device=DEV, dtype=torch.float64)
        face = torch.zeros(d.shape[0], device=DEV, dtype=torch.long)
        for b in range(self.lo.shape[0]):
            t1, t2 = (self.lo[b] - o) / d, (self.hi[b] - o) / d
            tn, an = torch.minimum(t1, t2).max(1)
            tf, af = torch.maximum(t1, t2).min(1)
            t, ax, ok = (tf, af, tf > 0) if b == 0 else (tn, an, (tn <= tf) & (tn > 0))
            up = (d.gather(1, ax[:, None])[:, 0] > 0) == (b == 0)
            hit = ok & (t < best)
            best = torch.where(hit, t, best)
            face = torch.where(hit, b * 6 + ax * 2 + up, face)
        pts, ax = o + best[:, None] * d, (face // 2) % 3
        uv = pts.gather(1, torch.stack([(ax == 0).long(), 2 - (ax == 2).long()], 1))
        k, phi = self.tex
        col = 0.5 + 0.5 * torch.sin(2 * np.pi * (k[face] * uv[:, None, :]).sum(-1) + phi[face])
        depth = best * (1 + 0.01 * torch.randn(best.shape, generator=gen, device=DEV, dtype=torch.float64))
        depth = torch.where((depth >= 0.5) & (depth <= 5.0), depth, torch.zeros_like(depth))
        return depth.reshape(H, W), col.reshape(H, W, 3), ray

    def frame(self, T, n, gen):
        """n points of one VGA frame: pixels of high intensity gradient, or any for a dense frame."""
        depth, col, ray = self.render(T, 640, 480, gen)
        gy, gx = torch.gradient(col[..., 2])
        mag, ok = torch.hypot(gx, gy).reshape(-1), depth.reshape(-1) > 0
        keep = ok & (mag > torch.quantile(mag[ok], 0.8)) if n <= 30000 else ok
        idx = keep.nonzero()[:, 0]
        while idx.numel() < n:   # a frame with few valid pixels: some pixels twice
            idx = torch.cat([idx, idx])
        idx = idx[torch.randperm(idx.numel(), generator=gen, device=DEV)[:n]].sort().values
        feat = torch.cat([col.reshape(-1, 3), (gx / 0.05).clamp(-1, 1).reshape(-1, 1),
                          (gy / 0.05).clamp(-1, 1).reshape(-1, 1)], 1)
        return depth.reshape(-1)[idx, None] * ray[idx], feat[idx]


def _dims(feat, dim):
    """The feature vectors cut or widened to `dim` columns."""
    return torch.cat([feat, feat[:, :3] * feat[:, 1:4]], 1)[:, :dim] if dim else None


def _rngs(seed):
    return np.random.default_rng(seed), torch.Generator(device=DEV).manual_seed(seed)


def _pair(scene, n, m, dim, seed, deg=3.0, metres=0.03):
    """Target and source clouds (float32 on the GPU) and the pose that maps the source onto the target."""
    rng, gen = _rngs(seed)
    if scene == "room":
        room = _Room(rng)
        P = _rigid(rng, deg, metres)
        (X, FX), (Z, FZ) = room.frame(room.T, n, gen), room.frame(room.T @ P, m, gen)
    else:
        tex = _textures(rng, 3)
        (X, FX), (Z, FZ) = _planes(tex, n, gen), _planes(tex, m, gen)
        P = _rigid(rng, deg, metres)
        Z = _move(np.linalg.inv(P), Z)
    f32 = [None if v is None else v.float().contiguous() for v in (X, _dims(FX, dim), Z, _dims(FZ, dim))]
    return (*f32, P)


def _near(P, seed):
    """A pose two degrees and two centimetres off P, as a motion model predicts it."""
    return _rigid(np.random.default_rng(seed + 77), 2.0, 0.02) @ P


def _uneven(case, count, seed):
    rng = random.Random(seed)
    return [(rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"]), rng.uniform(0.5, 5.0),
             rng.uniform(0.005, 0.05), rng.uniform(0.12, 0.18)) for _ in range(count)]


# ---- the calls -------------------------------------------------------------------------------

def _options(case):
    return {"feat_dim": case["dim"], "color_mode": MODES[case["mode"]], "color_scale": 1.0,
            "feat_bf16": case.get("bf16", 0)}


def _host(*arrays):
    return [None if a is None else a.cpu().numpy() for a in arrays]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "frontend":
        rng, gen = _rngs(seed)
        room, W, H = _Room(rng), case["width"], case["height"]
        depth, hsv, _ = room.render(room.T, W, H, gen)
        f = 525.0 * W / 640.0
        prm = cvo.cvo_frontend_params_default(fx=f, fy=f, cx=(W - 1) / 2, cy=(H - 1) / 2,
                                              percentile=case["percentile"], max_points=case["max_points"])
        out = [torch.zeros(W * H, c, device=DEV) for c in (3, 5)] + [torch.zeros(W * H, device=DEV, dtype=torch.int32)]
        return {"kind": kind, "ctx": cvo.Context(), "depth": depth.float().contiguous(),
                "hsv": hsv.float().contiguous(), "prm": prm, "out": out}
    if kind == "static":
        X, FX, Z, FZ, P = _pair("planes", case["n"], case["m"], case["dim"], seed)
        prm = cvo.cvo_params_default()
        for k, v in _options(case).items():
            setattr(prm, k, v)
        return {"kind": kind, "args": (X, FX, Z, FZ, prm, _near(P, seed), case["ell"]),
                "out": torch.empty(8, device=DEV, dtype=torch.float64)}
    s = {"kind": kind, "ctx": cvo.Context(**_options(case))}
    if kind == "batch":
        hx, hz, ells = [], [], []
        for i, (n, m, deg, metres, ell) in enumerate(_uneven(case, case["pairs"], seed)):
            X, FX, Z, FZ, _ = _pair("planes", n, m, case["dim"], seed * 4099 + i, deg, metres)
            torch.cuda.synchronize()
            hx.append(s["ctx"].set_cloud(X, FX))
            hz.append(s["ctx"].set_cloud(Z, FZ))
            ells.append(ell)
        s["batch"] = s["ctx"].batch(hx, hz, ell0=ells)
        s["P0"] = np.tile(np.eye(4), (case["pairs"], 1, 1))
    elif kind == "serve":
        sizes = _uneven(case, case["requests"], seed)
        s["keys"], s["frames"] = [], []
        for c in range(case["cameras"]):
            rng, gen = _rngs(seed * 4099 + c)
            tex = _textures(rng, 3)
            X, FX = _planes(tex, sizes[c][0], gen)
            FX = _dims(FX, case["dim"])
            torch.cuda.synchronize()
            s["keys"].append(s["ctx"].set_cloud(*_host(X.float(), None if FX is None else FX.float())))
            for n, _, deg, metres, _ in sizes[c::case["cameras"]]:
                Z, FZ = _planes(tex, n, gen)
                Z, FZ = _move(_rigid(rng, 0.6 * deg, 0.6 * metres), Z), _dims(FZ, case["dim"])
                s["frames"].append((s["keys"][c], *_host(Z.float(), None if FZ is None else FZ.float())))
    else:
        X, FX, Z, FZ, P = _pair(case["scene"], case["n"], case["m"], case["dim"], seed)
        torch.cuda.synchronize()
        s["target"] = s["ctx"].set_cloud(X, FX)
        if kind == "track":
            s["frame"] = _host(Z, FZ)
        else:
            s["source"] = s["ctx"].set_cloud(Z, FZ)
        if kind == "eval":
            s["P"], s["ell"] = _near(P, seed), case["ell"]
    return s


def _solved(P, stats):
    """Poses and last F of solves. The iteration at which the stop rule fires, and the counts that
    follow from it, hang on the last bits of a step length, so they are no result to compare."""
    return {"P": np.asarray(P, np.float32), "F": np.asarray([t["F_last"] for t in stats], np.float32)}


def run(state):
    kind = state["kind"]
    if kind == "static":
        out = state["out"]
        cvo.cvo_eval_gradient_static(*state["args"], out)
        sums = out.float()
        return {"F": sums[0], "grad6": sums[1:7], "pairs": out[7:]}
    ctx = state["ctx"]
    if kind == "frontend":
        xyz, feat, pixel = state["out"]
        n = ctx.frontend_select(state["depth"], state["hsv"], state["prm"], xyz, feat, pixel)
        return {"n": n, "xyz": xyz, "feat": feat, "pixel": pixel}   # zeros past the n points
    if kind == "eval":
        r = ctx.eval(state["target"], state["source"], state["P"], state["ell"])
        # the step model in lengthscales along the gradient: S_m (ell / |xi|)^m
        unit = state["ell"] / max(np.linalg.norm(r["grad6"]), 1e-300)
        return {"F": np.float32(r["F"]), "grad6": np.float32(r["grad6"]),
                "model": np.float32(r["S"] * unit ** np.arange(5)), "nnz": r["nnz"]}
    if kind == "align":
        P, st = ctx.align(state["target"], state["source"])
        return _solved(P, [st])
    if kind == "track":
        h = ctx.set_cloud(*state["frame"])
        P, st = ctx.align(state["target"], h)
        ctx.release(h)
        return _solved(P, [st])
    if kind == "batch":
        return _solved(*state["batch"].run(state["P0"]))
    tickets = [ctx.submit(key, Z, FZ) for key, Z, FZ in state["frames"]]
    done = {}
    while len(done) < len(tickets):
        for t in tickets:
            if t not in done:
                r = ctx.poll(t)
                if r is not None:
                    done[t] = r
        time.sleep(1e-4)
    return _solved([done[t][0] for t in tickets], [done[t][1] for t in tickets])


def work(case):
    """Bytes: inputs and outputs once. Operations: 44 per kept pair in a gradient pass and 104 in a
    step pass (22 and 52 FP32 instructions), pairs estimated from the density of the scene's surfaces."""
    kind = case["kind"]
    if kind == "frontend":
        n = case["width"] * case["height"]
        kept = n * (1 - case["percentile"] / 100)
        kept = min(kept, case["max_points"]) if case["max_points"] else kept
        return {"bytes": 16 * n + 36 * kept, "flops": 20 * n}
    point = 12 + 4 * case["dim"]
    area = 12.0 if case.get("scene") != "room" else 25.0
    kcut = 2 * math.log(1e3)

    def kept(n, m, ell):
        return m * min(n, n / area * math.pi * kcut * ell * ell)

    def solve(n, m, ell0, floor_iters):
        ells, e = [], ell0
        while e > 0.02:
            ells.append(e)
            e *= 0.9
        return 148 * sum(kept(n, m, e) for e in ells + [0.02] * floor_iters)

    if kind == "static":   # every pair is tested: 8 operations
        n, m = case["n"], case["m"]
        return {"bytes": (n + m) * point + 64, "flops": 8 * n * m + 44 * kept(n, m, case["ell"])}
    if kind == "eval":
        n, m = case["n"], case["m"]
        return {"bytes": (n + m) * point, "flops": 148 * kept(n, m, case["ell"])}
    if kind in ("align", "track"):
        n, m = case["n"], case["m"]
        return {"bytes": (n + m) * point, "flops": solve(n, m, 0.15, 130 if case["scene"] == "room" else 25)}
    count = case["pairs"] if kind == "batch" else case["requests"]
    n = (case["lo"] + case["hi"]) / 2
    return {"bytes": 2 * n * count * point, "flops": count * solve(n, n, 0.15, 25)}


# ---- the same results in 64 bits --------------------------------------------------------------

def _kept_pairs(X, Zt, rc2):
    """Index pairs within the cutoff, tested in 64 bits (a wider FP32 test finds the candidates)."""
    x, z = X.float(), Zt.float()
    rows = max(1, 60_000_000 // x.shape[0])
    for j0 in range(0, z.shape[0], rows):
        d2 = sum((x[None, :, a] - z[j0:j0 + rows, None, a]) ** 2 for a in range(3))
        for part in (d2 <= rc2 * 1.001 + 1e-5).nonzero().split(10_000_000):
            j, i = part[:, 0] + j0, part[:, 1]
            on = ((X[i] - Zt[j]) ** 2).sum(1) <= rc2
            yield i[on], j[on]


def _exact_sums(X, FX, Z, FZ, P, ell, mode, xi=None):
    """F and the gradient (or, with a direction, the five step sums along it) in FP64."""
    X, Z = X.double(), _move(P, Z.double())
    feats = None if FX is None or mode == NONE else (FX.double(), FZ.double())
    rc2 = 2 * ell * ell * math.log(1e3)
    total = torch.zeros(7 if xi is None else 5, device=DEV, dtype=torch.float64)
    for i, j in _kept_pairs(X, Z, rc2):
        e, z = X[i] - Z[j], Z[j]
        w = torch.exp(-(e * e).sum(1) / (2 * ell * ell))
        if feats is not None:
            f, g = feats[0][i], feats[1][j]
            w = w * ((f * g).sum(1) if mode == DOT else torch.exp(-((f - g) ** 2).sum(1) / (2 * 0.1 ** 2)))
        if xi is None:
            total += torch.cat([w.sum()[None], (w[:, None] * torch.linalg.cross(z, e)).sum(0) / ell ** 2,
                                (w[:, None] * e).sum(0) / ell ** 2])
            continue
        om = xi[:3].expand_as(z)
        u1 = torch.linalg.cross(om, z) + xi[3:]
        u2 = torch.linalg.cross(om, u1)
        u3 = torch.linalg.cross(om, u2)
        u4 = torch.linalg.cross(om, u3)

        def dot(a, b):
            return (a * b).sum(1)

        b = dot(e, u1) / ell ** 2
        c = (dot(e, u2) - dot(u1, u1)) / (2 * ell ** 2)
        d = (dot(e, u3) / 6 - dot(u1, u2) / 2) / ell ** 2
        h = (dot(e, u4) / 24 - dot(u1, u3) / 6 - dot(u2, u2) / 8) / ell ** 2
        terms = (torch.ones_like(b), b, b * b / 2 + c, b ** 3 / 6 + b * c + d,
                 b ** 4 / 24 + b * b * c / 2 + c * c / 2 + b * d + h)
        total += torch.stack([(w * t).sum() for t in terms])
    return total


def exact(case, seed):
    """None for whole solves: their last iteration is where the stop rule happens to fire."""
    kind = case["kind"]
    if kind in ("static", "eval"):
        X, FX, Z, FZ, P = _pair(case.get("scene", "planes"), case["n"], case["m"], case["dim"], seed)
        args = (X, FX, Z, FZ, _near(P, seed), case["ell"], case["mode"])
        g = _exact_sums(*args)
        if kind == "static":
            return {"F": g[0], "grad6": g[1:], "pairs": None}
        S = _exact_sums(*args, g[1:] / g[1:].norm())
        return {"F": g[0], "grad6": g[1:], "model": S * case["ell"] ** torch.arange(5, device=DEV), "nnz": None}
    if kind != "frontend":
        return None
    s = prepare(case, seed)
    depth, hsv, prm = s["depth"], s["hsv"], s["prm"]
    H, W = depth.shape
    # the selection is made on FP32 gradients, one rounding per operation
    gy, gx = torch.gradient(hsv[..., 2])
    mag, ok = torch.sqrt(gx * gx + gy * gy).double().reshape(-1), depth.reshape(-1) > 0
    keep = (ok & (mag > torch.quantile(mag[ok], prm.percentile / 100))).nonzero()[:, 0]
    if 0 < prm.max_points < keep.numel():
        keep = keep[torch.arange(prm.max_points, device=DEV) * keep.numel() // prm.max_points]
    z, u, v = depth.reshape(-1)[keep].double(), (keep % W).double(), (keep // W).double()
    xyz = torch.stack([(u - prm.cx) / prm.fx * z, (v - prm.cy) / prm.fy * z, z], 1)
    slope = (torch.stack([gx, gy], -1).reshape(-1, 2)[keep].double() / prm.grad_scale).clamp(-1, 1)
    out = torch.zeros(H * W, 8, device=DEV, dtype=torch.float64)
    out[:keep.numel()] = torch.cat([xyz, hsv.reshape(-1, 3)[keep].double(), slope], 1)
    return {"n": None, "xyz": out[:, :3].contiguous(), "feat": out[:, 3:].contiguous(), "pixel": None}

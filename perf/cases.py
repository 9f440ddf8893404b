"""Measured cases of the densification library, through its public entry points.

Each case is one call (or the short sequence of calls) that a SLAM system makes
per keyframe: densify a keyframe, densify a batch or a request queue of them,
start from the previous keyframe's planes, drive the steps by hand, score
given planes, then filter, median-filter and fuse the depth maps. Sizes are
the paper's online mode (1920x960) and the library's other workload sizes;
images come from a seeded ray caster below (a textured room with spheres and
boxes, seen from a short camera walk), depth maps from its ranges with the
noise, outliers and holes that densified maps show.
"""
import math

import numpy as np
import torch

import paper_2211_16266_gb300 as pm

DEV = "cuda:0"
ROOM = (2.0, 1.25, 1.5)  # half extents of the room in metres (x, y down, z)
DTYPES = {"u8": torch.uint8, "f16": torch.float16, "f32": torch.float32}
VIEW_SAMPLE_OPS = 55  # FP32 operations of one view-sample: transform, projection, interpolation, sums


# ------------------------------------------------------------------ the cases

def _densify(name, W, H, S, fmt, path="densify", **kw):
    c = dict(name=name, path=path, W=W, H=H, S=S, fmt=fmt, patch_w=11, stride=2, iters=8, best_k=min(3, S), weights=True,
             table=0, noise=0.0, host=False, n=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest keyframe in use (previews, tests): 2 sources, dense 7x7 window, no bilateral weights
        _densify("densify_256x128_u8", 256, 128, 2, "u8", patch_w=7, stride=1, iters=4, best_k=1, weights=False),
        # a half-size keyframe handed over and back in host memory, as a caller without CUDA does
        _densify("densify_960x480_f16_host", 960, 480, 6, "f16", host=True),
        # the paper's online resolution: one uint8 keyframe, 6 neighbours, then the consistency filter
        _densify("keyframe_1920x960_u8", 1920, 960, 6, "u8", path="keyframe", n=4),
        # quality mode: the largest keyframe, sensor noise, fp16 storage
        _densify("densify_3840x1920_f16", 3840, 1920, 8, "f16", noise=2.0),
        # a few iterations from the previous keyframe's warped planes, at a size that fills no tile
        _densify("warped_1000x502_f32", 1000, 502, 5, "f32", path="warped", iters=3),
        # initialisation and half-sweeps called one by one, ragged size, another window and neighbour table
        _densify("steps_250x130_f32", 250, 130, 3, "f32", path="steps", patch_w=9, stride=3, iters=3, best_k=2, table=1),
        # the matching cost of given planes (re-scoring a map, parity checks)
        _densify("cost_1920x960_u8", 1920, 960, 6, "u8", path="cost"),
        # keyframes of mixed size and view count in one captured batch
        _densify("batch_mixed_f16", 1920, 960, 4, "f16", path="batch", n=5),
        # a burst of requests against the frame ring: push, submit, wait
        _densify("serve_burst_f16", 960, 480, 6, "f16", path="serve", iters=4, n=6),
        # post-processing of the online pipeline at its resolution: filter, median, fusion with completeness
        dict(name="filter_1920x960x4", path="filter", W=1920, H=960, n=4),
        dict(name="median_1920x960_r2", path="median", W=1920, H=960, radius=2),
        dict(name="fuse_1920x960x6", path="fuse", W=1920, H=960, n=6, voxel=0.02),
    ]


def _even(rng, lo, hi):
    return 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)


def draw(rng):
    path = rng.choice(["densify", "densify", "densify", "keyframe", "warped", "steps", "cost", "batch", "serve", "filter",
                       "median", "fuse"])
    W = _even(rng, 64, 2600)
    H = max(16, 2 * round(W * rng.uniform(0.4, 0.6) / 2))
    if path in ("filter", "median"):  # the post-filters take any size, odd ones too
        W, H = W + rng.randrange(2), H + rng.randrange(2)
    if path == "filter":
        return dict(path=path, W=W, H=H, n=rng.randint(1, 8))
    if path == "median":
        return dict(path=path, W=W, H=H, radius=rng.randint(1, 3))
    if path == "fuse":
        return dict(path=path, W=W, H=H, n=rng.randint(1, 8), voxel=rng.choice([0.01, 0.02, 0.05]))
    if path in ("batch", "serve"):
        W, H = min(W, 960), min(H, 480)
    S = rng.randint(1, 10) if path != "batch" else rng.randint(2, 5)
    patch_w, stride = rng.choice([(11, 2), (11, 2), (7, 1), (5, 1), (9, 3), (9, 2), (13, 2)])
    c = _densify("", W, H, S, rng.choice(["u8", "f16", "f32"]), path=path, patch_w=patch_w, stride=stride,
                 iters=rng.randint(1, 8), best_k=rng.randint(1, S), weights=rng.random() < 0.75, table=rng.randrange(2),
                 noise=rng.choice([0.0, 0.0, 2.0]), host=path == "densify" and rng.random() < 0.25,
                 n=rng.randint(2, 5) if path in ("batch", "serve", "keyframe") else 1)
    del c["name"]
    # no more work than the largest keyframe above
    most = 3840 * 1920 * 8 * 36 * 8
    while c["W"] * c["H"] * c["S"] * _samples(c) * max(1, c["iters"]) * c["n"] > most:
        c["W"], c["H"] = max(64, 2 * (c["W"] // 3)), max(16, 2 * (c["H"] // 3))
    return c


def _samples(c):
    return ((c["patch_w"] - 1) // c["stride"] + 1) ** 2


def _params(c, key=0, **kw):
    s = dict(sigma_color=0.2, sigma_space=3.0) if c["weights"] else dict(sigma_color=0.0, sigma_space=0.0)
    p = dict(d_min=0.3, d_max=10.0, patch_w=c["patch_w"], patch_stride=c["stride"], iterations=c["iters"], best_k=c["best_k"],
             n_refine=6, neighbor_table=c["table"], seed=42, keyframe_id=key, **s)
    p.update(kw)
    return pm.pmsp_default_params(**p)


# ------------------------------------------------------------------ the scene

def _rotation(yaw, pitch, roll):
    c, s = math.cos, math.sin
    ry = np.array([[c(yaw), 0, s(yaw)], [0, 1, 0], [-s(yaw), 0, c(yaw)]])
    rx = np.array([[1, 0, 0], [0, c(pitch), -s(pitch)], [0, s(pitch), c(pitch)]])
    rz = np.array([[c(roll), -s(roll), 0], [s(roll), c(roll), 0], [0, 0, 1]])
    return ry @ rx @ rz


class _Scene:
    """A textured room with spheres and boxes, and a smooth camera walk of `n` poses through it."""

    def __init__(self, seed, n, objects=12):
        rng = np.random.default_rng(seed)
        half = np.array(ROOM)
        lim = np.array([1.4, 0.4, 0.9])
        pos, head, yaw = rng.uniform(-lim, lim), rng.uniform(0, 2 * math.pi), rng.uniform(-math.pi, math.pi)
        self.poses, centres = [], []
        for _ in range(n):
            R_cw = _rotation(yaw, math.radians(rng.normal(0, 2.0)), math.radians(rng.normal(0, 2.0)))
            self.poses.append((R_cw.T.copy(), -R_cw.T @ pos))
            centres.append(pos.copy())
            step = float(np.clip(rng.normal(0.15, 0.03), 0.08, 0.25))
            head += rng.normal(0, 0.35)
            d = np.array([math.sin(head), rng.normal(0, 0.1), math.cos(head)])
            nxt = pos + step * d / np.linalg.norm(d)
            if np.any(np.abs(nxt) > lim):
                head += math.pi / 2
            pos = np.clip(nxt, -lim, lim)
            yaw += math.radians(rng.uniform(-10, 10))
        self.objects = []
        for i in range(objects):
            r = float(rng.uniform(0.2, 0.7))
            for _ in range(60):
                c = rng.uniform(-half, half)
                if min(np.max(np.abs(c - p)) for p in centres) > r + 0.3 and min(np.linalg.norm(c - p) for p in centres) > r + 0.3:
                    self.objects.append((i % 2, c, r))
                    break
        gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 11)
        self.noise = torch.rand(64, 64, 64, generator=gen, device=DEV).reshape(-1)

    def _dirs(self, R, W, H, ss, v0, v1):
        u = (torch.arange(W * ss, device=DEV, dtype=torch.float64) + 0.5) / ss
        v = (torch.arange(v0 * ss, v1 * ss, device=DEV, dtype=torch.float64) + 0.5) / ss
        lon, lat = (2 * math.pi / W) * u - math.pi, math.pi / 2 - (math.pi / H) * v
        d = torch.stack([torch.cos(lat)[:, None] * torch.sin(lon), (-torch.sin(lat))[:, None].expand(-1, W * ss),
                         torch.cos(lat)[:, None] * torch.cos(lon)])
        return torch.einsum("ji,jhw->ihw", torch.tensor(R, device=DEV), d).float()  # world frame: R^T d

    def _trace(self, o, d):
        """Range, world normal and object number along unit directions d (3, h, w) from o."""
        half = torch.tensor(ROOM, device=DEV)
        t_ax = (torch.sign(d) * half[:, None, None] - o[:, None, None]) / torch.where(d == 0, torch.full_like(d, 1e-12), d)
        t, ax = t_ax.min(0)
        n = -torch.sign(d) * (torch.arange(3, device=DEV)[:, None, None] == ax)
        which = torch.zeros_like(ax)
        for i, (kind, c, r) in enumerate(self.objects):
            oc = o - torch.tensor(c, device=DEV, dtype=torch.float32)
            if kind == 0:
                b, q = (d * oc[:, None, None]).sum(0), float((oc * oc).sum()) - r * r
                disc = b * b - q
                ti = torch.where(disc > 0, -b - disc.clamp_min(0).sqrt(), torch.full_like(b, 1e9))
                ni = (oc[:, None, None] + ti * d) / r
            else:
                inv = 1.0 / torch.where(d == 0, torch.full_like(d, 1e-12), d)
                a1, a2 = (-r - oc[:, None, None]) * inv, (r - oc[:, None, None]) * inv
                near, k = torch.minimum(a1, a2).max(0)
                far = torch.maximum(a1, a2).min(0)[0]
                ti = torch.where(near <= far, near, torch.full_like(near, 1e9))
                ni = -torch.sign(d) * (torch.arange(3, device=DEV)[:, None, None] == k)
            hit = (ti > 1e-6) & (ti < t)
            t, n, which = torch.where(hit, ti, t), torch.where(hit, ni, n), torch.where(hit, i + 1, which)
        return t, n, which

    def _albedo(self, p, which):
        """Four octaves of value noise (3 cycles per metre and up) on DN 30 to 220."""
        total, amp, freq = 0.0, 1.0, 3.0
        for octave in range(4):
            x = p * freq + (which * 7.31 + octave * 17.7)
            i = torch.floor(x)
            f = x - i
            f = f * f * (3 - 2 * f)
            i = i.to(torch.int64)
            for corner in range(8):
                w, at = 1.0, 0
                for a in range(3):
                    b = (corner >> a) & 1
                    w = w * (f[a] if b else 1 - f[a])
                    at = at * 64 + ((i[a] + b) & 63)
                total = total + amp * w * self.noise[at]
            amp, freq = amp / 2, freq * 2
        return 30.0 + 190.0 * total / 1.875

    def image(self, k, W, H, fmt, noise=0.0, seed=0):
        """Panorama of pose k, 2x2 supersampled, as the library takes it."""
        R, t = self.poses[k]
        o = torch.tensor(-R.T @ t, device=DEV, dtype=torch.float32)
        rows = max(1, (1 << 20) // W)
        out = torch.empty(H, W, device=DEV)
        for v0 in range(0, H, rows):
            v1 = min(H, v0 + rows)
            d = self._dirs(R, W, H, 2, v0, v1)
            r, _, which = self._trace(o, d)
            out[v0:v1] = self._albedo(o[:, None, None] + r * d, which).reshape(v1 - v0, 2, W, 2).mean((1, 3))
        if noise:
            gen = torch.Generator(device=DEV).manual_seed(seed)
            out += noise * torch.randn(H, W, generator=gen, device=DEV)
        dn = out.clamp(0, 255)
        if fmt == "u8":
            return dn.round().to(torch.uint8)
        return (dn / 255.0 - (0.5 if fmt == "f16" else 0.0)).to(DTYPES[fmt])  # fp16 is stored centred on 0

    def planes(self, k, W, H):
        """Range (H, W) and normal (3, H, W) in the camera frame of pose k."""
        R, t = self.poses[k]
        o = torch.tensor(-R.T @ t, device=DEV, dtype=torch.float32)
        r, n, _ = self._trace(o, self._dirs(R, W, H, 1, 0, H))
        return r.contiguous(), torch.einsum("ij,jhw->ihw", torch.tensor(R, device=DEV, dtype=torch.float32), n).contiguous()

    def depth(self, k, W, H, seed, holes=0.0):
        """The range map of pose k as densification leaves it: 0.3 % noise, 8 % outliers in patches, and `holes` removed."""
        gen = torch.Generator(device=DEV).manual_seed(seed)
        rand = lambda *s: torch.rand(*s, generator=gen, device=DEV)  # noqa: E731
        r, _ = self.planes(k, W, H)
        r = r * (1 + 0.003 * torch.randn(H, W, generator=gen, device=DEV))
        coarse = torch.nn.functional.interpolate(rand(1, 1, H // 6 + 1, W // 6 + 1), size=(H, W))[0, 0]
        r = torch.where(coarse < 0.08, 1.0 / (0.1 + rand(H, W) * (1 / 0.3 - 0.1)), r)
        if holes:
            r = torch.where((coarse > 1 - holes) | (rand(H, W) < holes / 4), torch.zeros_like(r), r)
        return r.contiguous()


# ------------------------------------------------------------------ inputs

def _maps(W, H):
    return pm.Maps.empty(W, H, device=DEV)


def _problem(scene, at, c, W, H, S, seed):
    """(ref, ref_pose, srcs, src_poses): the middle one of S + 1 consecutive frames against the others."""
    frames = [(scene.image(at + k, W, H, c["fmt"], c["noise"], seed * 64 + at + k), scene.poses[at + k]) for k in range(S + 1)]
    if c["host"]:
        frames = [(im.cpu().numpy(), pose) for im, pose in frames]
    mid = S // 2
    rest = frames[:mid] + frames[mid + 1:]
    return frames[mid][0], frames[mid][1], [f[0] for f in rest], [f[1] for f in rest]


def _post(s, case, seed):
    W, H, n = case["W"], case["H"], case.get("n", 1)
    scene = _Scene(seed, max(n + 1, 6))
    if case["path"] == "filter":
        s["depth"], s["pose"] = scene.depth(n // 2, W, H, seed), scene.poses[n // 2]
        others = [k for k in range(n + 1) if k != n // 2]
        s["nbrs"] = [scene.depth(k, W, H, seed + 100 + k) for k in others]
        s["nbr_poses"] = [scene.poses[k] for k in others]
        s["out"], s["agree"] = torch.empty(H, W, device=DEV), torch.empty(H, W, device=DEV, dtype=torch.int32)
    elif case["path"] == "median":
        s["depth"] = scene.depth(0, W, H, seed, holes=0.2)
        s["out"] = torch.empty(H, W, device=DEV)
    else:
        s["depths"] = [scene.depth(k, W, H, seed + k, holes=0.2) for k in range(n)]
        s["poses"] = [scene.poses[k] for k in range(n)]
        s["hit"] = torch.empty(360, 720, device=DEV, dtype=torch.uint8)
        s["cloud"] = torch.zeros(W * H, 3, device=DEV)  # the map's point buffer and each point's origin
        s["origin"] = torch.zeros(W * H, device=DEV, dtype=torch.int64)
    return s


def prepare(case, seed):
    c, path = case, case["path"]
    s = {"case": c, "ctx": pm.Context(0)}
    if path in ("filter", "median", "fuse"):
        return _post(s, c, seed)
    W, H, S, n = c["W"], c["H"], c["S"], c["n"]
    if path == "batch":  # n keyframes of the size, half and a third of it, from S views on
        scene, probs = _Scene(seed, S + n + 2), []
        for k in range(n):
            w, h = 2 * (W // (2, 2, 1, 3, 2)[k % 5] // 2), 2 * (H // (2, 2, 1, 3, 2)[k % 5] // 2)
            sk = min(S + k, 10)
            p = dict(c, best_k=min(c["best_k"], sk))
            probs.append((*_problem(scene, k % 3, c, w, h, sk, seed), _params(p, key=k), _maps(w, h)))
        s["batch"] = pm.Batch(probs)
        s["tuning"] = pm.pmsp_tuning(0, 0, 0, 1, 0, 1, 0)
        return s
    if path == "serve":  # a ring of frames, n requests for consecutive keyframes, the last ones filtered
        m = S + n
        scene = _Scene(seed, m)
        s["frames"] = [(k, scene.image(k, W, H, c["fmt"], c["noise"], seed * 64 + k), scene.poses[k]) for k in range(m)]
        s["requests"] = []
        for k in range(n):
            at = k + S // 2
            near = [f for f in range(k, k + S + 1) if f != at]
            flt = [f for f in (at - 2, at - 1) if f >= S // 2] if k >= 2 else []
            s["requests"].append((at, near, _params(c, key=at), flt, _maps(W, H)))
        return s
    scene = _Scene(seed, max(S, n) + 1)
    s["problem"] = _problem(scene, 0, c, W, H, S, seed)
    s["params"] = _params(c, key=1)
    s["out"] = pm.Maps.empty(W, H) if c["host"] else _maps(W, H)
    mid = S // 2
    if path == "keyframe":  # the depth maps of n neighbours, densified before
        others = [k for k in range(n + 1) if k != mid][:n]
        s["nbrs"] = [scene.depth(k, W, H, seed + 100 + k) for k in others]
        s["nbr_poses"] = [scene.poses[k] for k in others]
        s["kept"], s["agree"] = torch.empty(H, W, device=DEV), torch.empty(H, W, device=DEV, dtype=torch.int32)
    elif path == "warped":  # the previous keyframe's finished maps
        k = mid - 1 if mid else mid + 1
        s["prev"] = pm.Maps(scene.depth(k, W, H, seed + 200), scene.planes(k, W, H)[1], torch.zeros(H, W, device=DEV))
        s["prev_pose"] = scene.poses[k]
    elif path == "cost":  # the planes of a map: the surfaces, with the noise of densification
        gen = torch.Generator(device=DEV).manual_seed(seed + 300)
        nrm = scene.planes(mid, W, H)[1] + 0.1 * torch.randn(3, H, W, generator=gen, device=DEV)
        s["out"].normal.copy_(nrm / nrm.norm(dim=0))
        s["out"].depth.copy_(scene.depth(mid, W, H, seed + 300))
    return s


# ------------------------------------------------------------------ one pass

def _of(m):
    return [m.depth, m.normal, m.cost]


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    path = c["path"]
    if path == "densify":
        return _of(pm.pmsp_densify(ctx, *s["problem"], s["params"], s["out"]))
    if path == "keyframe":
        m = pm.pmsp_densify(ctx, *s["problem"], s["params"], s["out"])
        pm.pmsp_consistency_filter(ctx, m.depth, s["problem"][1], s["nbrs"], s["nbr_poses"], out=s["kept"], agree=s["agree"])
        return _of(m) + [s["kept"], s["agree"]]
    if path == "warped":
        return _of(pm.pmsp_densify_warped(ctx, *s["problem"], s["params"], s["prev"], s["prev_pose"], s["out"]))
    if path == "steps":
        m = pm.pmsp_init(ctx, *s["problem"], s["params"], s["out"])
        for it in range(c["iters"]):
            for colour in range(2):
                pm.pmsp_halfsweep(ctx, *s["problem"], s["params"], colour, it, m)
        return _of(m)
    if path == "cost":
        return pm.pmsp_cost_map(ctx, *s["problem"], s["params"], s["out"]).cost
    if path == "batch":
        return [_of(m) for m in pm.pmsp_densify_batch(ctx, s["batch"], pm.PMSP_BATCH_GRAPH, s["tuning"])]
    if path == "serve":
        for k, im, pose in s["frames"]:
            pm.pmsp_ring_push(ctx, k, im, pose)
        tickets = [(pm.pmsp_submit(ctx, at, near, p, flt, min_views=1), out) for at, near, p, flt, out in s["requests"]]
        return [_of(pm.pmsp_wait(ctx, t, 60_000, out)) for t, out in tickets]
    if path == "filter":
        return list(pm.pmsp_consistency_filter(ctx, s["depth"], s["pose"], s["nbrs"], s["nbr_poses"], out=s["out"],
                                               agree=s["agree"]))
    if path == "median":
        return pm.pmsp_median_filter(ctx, s["depth"], radius=c["radius"], out=s["out"])
    points, src, count = pm.pmsp_fuse(ctx, s["depths"], s["poses"], voxel=c["voxel"])
    share, hit = pm.pmsp_completeness(ctx, points, s["poses"][0], hit=s["hit"])
    kept = min(count, len(s["cloud"]))
    s["cloud"][:kept] = points[:kept]
    s["origin"][:kept] = src[:kept]
    return [s["cloud"], s["origin"], count, share, hit]


# ------------------------------------------------------------------ what a pass cannot do without

def _densify_work(c, W, H, S):
    px, size = W * H, {"u8": 1, "f16": 2, "f32": 4}[c["fmt"]]
    evals = 1 if c["path"] == "cost" else 1 + 14 * c["iters"]
    return px * ((S + 1) * size + 20), px * evals * _samples(c) * S * VIEW_SAMPLE_OPS


def work(case):
    c, path = case, case["path"]
    px = c["W"] * c["H"]
    if path == "filter":
        return {"bytes": px * 4 * (c["n"] + 3), "flops": px * c["n"] * 70}
    if path == "median":
        return {"bytes": px * 8, "flops": px * 4 * (2 * c["radius"] + 1) ** 2}
    if path == "fuse":
        return {"bytes": px * 4 * c["n"] + 360 * 720, "flops": px * c["n"] * 25}
    if path == "batch":
        parts = []
        for k in range(c["n"]):
            f = (2, 2, 1, 3, 2)[k % 5]
            parts.append(_densify_work(c, 2 * (c["W"] // f // 2), 2 * (c["H"] // f // 2), min(c["S"] + k, 10)))
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    b, f = _densify_work(c, c["W"], c["H"], c["S"])
    if path == "serve":
        return {"bytes": c["n"] * b, "flops": c["n"] * f}
    if path == "keyframe":
        return {"bytes": b + px * 4 * (c["n"] + 2), "flops": f + px * c["n"] * 70}
    if path == "warped":
        return {"bytes": b + px * 16, "flops": f}
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit values

def _bearing(u, v, W, H):
    lon, lat = 2 * math.pi * (u + 0.5) / W - math.pi, math.pi / 2 - math.pi * (v + 0.5) / H
    return torch.stack([torch.cos(lat) * torch.sin(lon), -torch.sin(lat), torch.cos(lat) * torch.cos(lon)])


def _project(X, W, H):
    lon, lat = torch.atan2(X[0], X[2]), torch.atan2(-X[1], torch.hypot(X[0], X[2]))
    return W * (lon + math.pi) / (2 * math.pi) - 0.5, H * (math.pi / 2 - lat) / math.pi - 0.5


def _relative(a, b):
    """Pose from camera a to camera b."""
    R = b[0] @ a[0].T
    return torch.tensor(R, device=DEV), torch.tensor(b[1] - R @ a[1], device=DEV)


def _exact_cost(c, s):
    (ref, ref_pose, srcs, poses), W, H = s["problem"], c["W"], c["H"]
    scale = 255.0 if c["fmt"] == "u8" else 1.0
    ref = torch.as_tensor(ref, device=DEV).double() / scale
    srcs = [torch.as_tensor(x, device=DEV).double() / scale for x in srcs]
    r, st = (c["patch_w"] - 1) // 2, c["stride"]
    offs = [(a, b) for a in range(-r, r + 1, st) for b in range(-r, r + 1, st)]
    depth, normal = s["out"].depth.double(), s["out"].normal.double()
    out = torch.empty(H, W, device=DEV, dtype=torch.float64)
    u = torch.arange(W, device=DEV)
    for v0 in range(0, H, 64):
        v = torch.arange(v0, min(H, v0 + 64), device=DEV)
        vv, uu = v[:, None].expand(-1, W), u[None, :].expand(len(v), -1)
        n = normal[:, v0:v0 + 64]
        dn = depth[v0:v0 + 64] * (n * _bearing(uu.double(), vv.double(), W, H)).sum(0)
        Ip, valid = ref[vv, uu], torch.ones_like(dn, dtype=torch.bool)
        ws, Is, Xs = [], [], []
        for a, b in offs:
            qv, qu = (vv + a).clamp(0, H - 1), (uu + b) % W
            rq = _bearing(qu.double(), qv.double(), W, H)
            den = (n * rq).sum(0)
            valid &= den < -1e-6
            Iq, w = ref[qv, qu], torch.ones_like(dn)
            if c["weights"]:
                w = torch.exp(-(Iq - Ip) ** 2 / (2 * 0.2 ** 2) - (a * a + b * b) / (2 * 3.0 ** 2))
            ws.append(w), Is.append(Iq), Xs.append(dn / den * rq)
        w, I, X = torch.stack(ws), torch.stack(Is), torch.stack(Xs, 1)
        Sw, SI, SII = w.sum(0), (w * I).sum(0), (w * I * I).sum(0)
        varI, costs = Sw * SII - SI * SI, []
        for im, pose in zip(srcs, poses):
            R, t = _relative(ref_pose, pose)
            uc, vc = _project(torch.einsum("ij,jkhw->ikhw", R, X) + t[:, None, None, None], W, H)
            i, j = torch.floor(uc), torch.floor(vc)
            fx, fy = uc - i, vc - j
            i0, j0 = i.long() % W, j.long().clamp(0, H - 1)
            i1, j1 = (i.long() + 1) % W, (j.long() + 1).clamp(0, H - 1)
            J = (im[j0, i0] * (1 - fx) + im[j0, i1] * fx) * (1 - fy) + (im[j1, i0] * (1 - fx) + im[j1, i1] * fx) * fy
            SJ, SJJ, SIJ = (w * J).sum(0), (w * J * J).sum(0), (w * I * J).sum(0)
            varJ = Sw * SJJ - SJ * SJ
            ncc = ((Sw * SIJ - SI * SJ) / torch.sqrt((varI * varJ).clamp_min(1e-300))).clamp(-1, 1)
            bad = ~valid | (varI < 1e-8 * Sw * Sw) | (varJ < 1e-8 * Sw * Sw)
            costs.append(torch.where(bad, torch.full_like(ncc, 2.0), 1 - ncc))
        out[v0:v0 + 64] = torch.stack(costs).sort(0)[0][:c["best_k"]].mean(0)
    return out


def _exact_filter(c, s):
    W, H = c["W"], c["H"]
    v, u = torch.meshgrid(torch.arange(H, device=DEV), torch.arange(W, device=DEV), indexing="ij")
    d = s["depth"].double()
    X = d * _bearing(u.double(), v.double(), W, H)
    agree = torch.zeros(H, W, device=DEV, dtype=torch.int32)
    for nb, pose in zip(s["nbrs"], s["nbr_poses"]):
        R, t = _relative(s["pose"], pose)
        uc, vc = _project(torch.einsum("ij,jhw->ihw", R, X) + t[:, None, None], W, H)
        ui, vi = torch.floor(uc + 0.5).long() % W, torch.floor(vc + 0.5).long().clamp(0, H - 1)
        dj = nb.double()[vi, ui]
        Rb, tb = _relative(pose, s["pose"])
        Z = torch.einsum("ij,jhw->ihw", Rb, dj * _bearing(ui.double(), vi.double(), W, H)) + tb[:, None, None]
        u2, v2 = _project(Z, W, H)
        du = u2 - u
        du = du - W * torch.floor(du / W + 0.5)
        agree += ((d > 0) & (dj > 0) & (torch.hypot(du, v2 - v) < 1.0)).int()
    return [torch.where((d > 0) & (agree >= 2), d, torch.zeros_like(d)), None]


def _exact_median(c, s):
    W, H, r = c["W"], c["H"], c["radius"]
    d = s["depth"].double()
    padded = torch.nn.functional.pad(d, (0, 0, r, r))  # rows outside the panorama hold no value
    rows = [torch.roll(padded[a:a + H], -b, 1) for a in range(2 * r + 1) for b in range(-r, r + 1)]
    win = torch.stack(rows)
    count = (win > 0).sum(0)
    win = torch.where(win > 0, win, torch.full_like(win, math.inf)).sort(0)[0]
    m = win.gather(0, ((count - 1).clamp_min(0) // 2)[None])[0]
    off = (s["depth"] - m.float()).abs() > torch.tensor(0.05, device=DEV) * m.float()  # decided in FP32, as the maps are stored
    return torch.where((d > 0) & ~off, d, torch.zeros_like(d))


def exact(case, seed):
    path = case["path"]
    if path not in ("cost", "filter", "median"):
        return None  # the random search and the voxel map have no 64-bit value of their own
    s = prepare(case, seed)
    return {"cost": _exact_cost, "filter": _exact_filter, "median": _exact_median}[path](case, s)

"""Timed cases of the RKHS-BA library: what its users have it do, at the sizes they have.

A case names an operation of the public interface (paper_2403_01254_gb300.rkhsba)
and a scene.  Scenes are made on the GPU from the seed:

  rgbd    three walls and a sphere in a 10 m cube, RGB and one-hot classes
          (RGB-D frames, ell = 0.1 m, colour lengthscale 0.1)
  object  scans of one small asymmetric object (ell = 0.1), with or without
          part labels (multi-view registration, global initialisation)
  street  LiDAR scans along a street: ground, facades, boxes, poles, range
          noise; 19-class label distributions, FP32 or BF16 (ell = 0.3 m)
  loop    the same street walked in a 16 m loop, edges between near frames and
          between revisits (global mapping)

Operations:

  eval      loss, gradient, Gauss-Newton matrix and pair counts of a resident problem
  static    the same without device allocation (rkhsba_eval_static)
  solve     the LM solve from an initial guess, a fixed number of iterations
  step      device-resident stepping: grids rebuilt, poses set, LM iterations, state read
  fresh     a new problem each time: create from device arrays, evaluate, destroy
  search    the 60-rotation search of one frame against another
  distance  inner products, distances and cosines of every edge
  serve     requests through the batching server, from host arrays to poses

The pair arithmetic is FP32 (include/rkhsba.h) and the doubles that the library
hands out carry its rounding, so losses, gradients, matrices and poses are
passed on as FP32, the precision that they have; pair counts are whole numbers.
A solve's pair_terms is left out: it counts the pairs at poses that themselves
carry that rounding (the evaluations return their counts).
"""
import math

import numpy as np
import torch

import paper_2403_01254_gb300 as pk
from paper_2403_01254_gb300 import rkhsba as api

DEV = "cuda"


# ------------------------------------------------------------------- cases --
def _case(name, op, scene, frames, points, **kw):
    c = dict(name=name, op=op, scene=scene, frames=frames, points=points, bf16=False, classes=0, colour=False,
             top_k=0, sem_min=0.0, iters=0, unit_queries=32, requests=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: two RGB-D frames of ~2000 points (the paper's
        # downsampled frames), one evaluation
        _case("rgbd_eval_2x2000", "eval", "rgbd", 2, 2000, classes=5, colour=True),
        # the same pair registered: what an odometry front end calls per frame
        _case("rgbd_solve_2x2000", "solve", "rgbd", 2, 2000, classes=5, colour=True, iters=10),
        # a small window evaluated from inside another runtime, no allocation
        _case("rgbd_static_4x5003", "static", "rgbd", 4, 5003, classes=10, colour=True),
        # global initialisation of two object scans, part labels
        _case("object_search_2x4000", "search", "object", 2, 4000, classes=3),
        # multi-view registration without labels (plain kernel correlation)
        _case("object_plain_4x8000", "eval", "object", 4, 8000),
        # a window of dense RGB-D frames with colour and classes
        _case("rgbd_eval_5x20011", "eval", "rgbd", 5, 20011, classes=10, colour=True),
        # LiDAR multi-view registration, FP32 class distributions, all pairs
        _case("street_eval_8x20000", "eval", "street", 8, 20000, classes=19),
        # the same with the paper's eight neighbours per point
        _case("street_top8_8x20000", "eval", "street", 8, 20000, classes=19, top_k=8),
        # a loop-closure check: a new small problem, used once
        _case("street_fresh_4x30000", "fresh", "street", 4, 30000, classes=19, bf16=True),
        # sliding-window odometry: one step per new frame, BF16 labels
        _case("street_step_10x50000", "step", "street", 10, 50000, classes=19, bf16=True, iters=1),
        # a batch of requests through the server (2-6 frames, 5k-20k points each)
        _case("street_serve_6", "serve", "street", 6, 20000, classes=19, bf16=True, iters=6, requests=6),
        # global mapping, the largest problem one GPU is given, at the unit
        # size that rkhsba_autotune picks for it
        _case("loop_eval_64x100000", "eval", "loop", 64, 100000, classes=19, bf16=True, unit_queries=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rgbd", "rgbd", "object", "search", "street", "street", "variant", "fresh", "step",
                       "serve", "loop"])
    if kind == "rgbd":
        op = rng.choice(["eval", "eval", "solve", "static", "distance"])
        return _unnamed(op, "rgbd", rng.randint(2, 4 if op == "static" else 6),
                        _log_int(rng, 1000, 8000 if op == "static" else 30000), classes=rng.choice([0, 5, 10]),
                        colour=rng.random() < 0.8, iters=rng.randint(3, 12))
    if kind == "object":
        return _unnamed(rng.choice(["eval", "solve", "distance"]), "object", rng.randint(2, 5),
                        _log_int(rng, 1000, 8000), classes=rng.choice([0, 0, 3]), iters=rng.randint(3, 12))
    if kind == "search":
        return _unnamed("search", "object", 2, _log_int(rng, 1000, 8000), classes=rng.choice([0, 3]))
    if kind == "street":
        return _unnamed(rng.choice(["eval", "eval", "distance", "solve"]), "street", rng.randint(2, 9),
                        _log_int(rng, 5000, 100000), classes=rng.choice([4, 10, 19, 19, 28]),
                        bf16=rng.random() < 0.5, iters=rng.randint(2, 6))
    if kind == "variant":
        v = rng.choice(["top", "prune"])
        return _unnamed("eval", "street", rng.randint(2, 8), _log_int(rng, 5000, 40000), classes=19,
                        bf16=rng.random() < 0.5, top_k=rng.randint(1, 8) if v == "top" else 0,
                        sem_min=0.1 if v == "prune" else 0.0)
    if kind == "fresh":
        return _unnamed("fresh", rng.choice(["street", "rgbd"]), rng.randint(2, 6), _log_int(rng, 2000, 60000),
                        classes=10, bf16=rng.random() < 0.5)
    if kind == "step":
        return _unnamed("step", "street", rng.randint(3, 10), _log_int(rng, 10000, 80000), classes=19,
                        bf16=rng.random() < 0.7, iters=rng.randint(1, 3))
    if kind == "serve":
        return _unnamed("serve", "street", rng.randint(2, 6), _log_int(rng, 5000, 20000), classes=19, bf16=True,
                        iters=rng.randint(3, 8), requests=rng.randint(2, 8))
    return _unnamed("eval", "loop", rng.randint(6, 20), _log_int(rng, 40000, 100000), classes=19, bf16=True,
                    unit_queries=rng.choice([32, 64]))


def _unnamed(*a, **kw):
    c = _case("", *a, **kw)
    del c["name"]
    if c["op"] not in ("solve", "step", "serve"):
        c["iters"] = 0
    return c


# ------------------------------------------------------------------ scenes --
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)


def _rotation(axis, angle):
    axis = np.asarray(axis, np.float64) / np.linalg.norm(axis)
    w, (x, y, z) = math.cos(angle / 2), math.sin(angle / 2) * axis
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _pose(R, t):
    T = np.eye(4)
    T[:3, :3], T[:3, 3] = R, t
    return T


def _random_pose(rng, max_deg, max_trans):
    u = rng.normal(size=3)
    return _pose(_rotation(rng.normal(size=3), math.radians(rng.uniform(0.2, 1.0) * max_deg)),
                 rng.uniform(0.2, 1.0) * max_trans * u / np.linalg.norm(u))


def _to_local(pts, T):
    T = torch.tensor(T, device=DEV)
    return (pts - T[:3, 3]) @ T[:3, :3]


def _labels(g, cls, classes, bf16):
    """Class distributions close to Dirichlet(0.3 + 10 e_class); BF16 values when bf16."""
    n = len(cls)
    p = _rand(g, n, classes).pow_(1 / 0.3)
    p.mul_(-torch.log(_rand(g, n, classes).clamp_(min=1e-12)))
    p[torch.arange(n, device=DEV), cls % classes] += (10.0 + 3.2 * _randn(g, n)).clamp_(min=3.0)
    p = (p / p.sum(1, keepdim=True)).float()
    return p.bfloat16().float() if bf16 else p


def _all_pairs(K):
    return [(a, b) for a in range(K) for b in range(a + 1, K)]


def _rgbd_scene(case, seed):
    g, rng = _gen(seed), np.random.default_rng(seed)
    K, n = case["frames"], case["points"]
    colours = torch.tensor([[0.55, 0.45, 0.35], [0.80, 0.80, 0.75], [0.30, 0.45, 0.70], [0.85, 0.20, 0.15]],
                           device=DEV, dtype=torch.float64)
    share = torch.tensor([100.0, 100.0, 100.0, 4 * math.pi * 1.5 ** 2], device=DEV, dtype=torch.float64)
    edges_p = torch.cumsum(share / share.sum(), 0)
    gt = [np.eye(4)] + [_random_pose(rng, 10.0, 0.3) for _ in range(K - 1)]
    xyz, sem, rgb = [], [], []
    for m in range(K):
        prim = torch.searchsorted(edges_p, _rand(g, n)).clamp_(max=3)
        u = 10.0 * _rand(g, n, 2)
        v = _randn(g, n, 3)
        v = v / v.norm(dim=1, keepdim=True)
        zero = torch.zeros(n, device=DEV, dtype=torch.float64)
        flat = torch.stack([torch.stack([u[:, 0], u[:, 1], zero], 1), torch.stack([zero, u[:, 0], u[:, 1]], 1),
                            torch.stack([u[:, 0], zero, u[:, 1]], 1),
                            torch.tensor([5.0, 5.0, 3.0], device=DEV, dtype=torch.float64) + 1.5 * v])
        pts = flat[prim, torch.arange(n, device=DEV)] + 0.01 * _randn(g, n, 3)
        xyz.append(_to_local(pts, gt[m]))
        if case["classes"]:
            sem.append(torch.nn.functional.one_hot(prim, max(4, case["classes"]))[:, :case["classes"]].float())
        if case["colour"]:
            rgb.append((colours[prim] + 0.02 * _randn(g, n, 3)).clamp_(0, 1).float())
    init = [gt[0]] + [T @ _random_pose(rng, 3.0, 0.1) for T in gt[1:]]
    return dict(xyz=xyz, sem=sem or None, rgb=rgb or None, edges=_all_pairs(K), poses=np.stack(init), ell=0.1,
                ell_color=0.1 if case["colour"] else 0.0)


def _object_scene(case, seed):
    g, rng = _gen(seed), np.random.default_rng(seed)
    K, n = case["frames"], case["points"]
    dd = dict(device=DEV, dtype=torch.float64)
    gt = [np.eye(4)] + [_random_pose(rng, 90.0, 0.5) for _ in range(K - 1)]
    xyz, sem = [], []
    d = torch.tensor([-1.0, 0.3, 0.5], **dd)
    d = d / d.norm()
    u1 = torch.linalg.cross(d, torch.tensor([0.0, 0.0, 1.0], **dd))
    u1 = u1 / u1.norm()
    u2 = torch.linalg.cross(d, u1)
    rad = torch.tensor([0.4, 0.25, 0.15], **dd)
    for m in range(K):
        prim = torch.searchsorted(torch.tensor([0.59, 0.85], **dd), _rand(g, n))
        v = _randn(g, n, 3)
        v = v / v.norm(dim=1, keepdim=True)
        nb = v / rad
        nb = nb / nb.norm(dim=1, keepdim=True)
        face = (6 * _rand(g, n)).long().clamp_(max=5)
        cube = 0.25 * _rand(g, n, 3) - 0.125
        sgn = torch.where(face % 2 == 0, 1.0, -1.0).double()
        nc = torch.nn.functional.one_hot(face // 2, 3).double() * sgn[:, None]
        cube = torch.where(nc != 0, 0.125 * nc, cube) + torch.tensor([0.45, 0.2, 0.12], **dd)
        th, s = 2 * math.pi * _rand(g, n, 1), 0.6 * _rand(g, n, 1)
        nt = torch.cos(th) * u1 + torch.sin(th) * u2
        tail = torch.tensor([-0.35, 0.0, 0.0], **dd) + s * d + 0.06 * nt
        at = torch.arange(n, device=DEV)
        pts = torch.stack([v * rad, cube, tail])[prim, at]
        nrm = torch.stack([nb, nc, nt])[prim, at]
        xyz.append(_to_local(pts + 0.01 * _randn(g, n, 1) * nrm, gt[m]))
        if case["classes"]:
            sem.append(_labels(g, prim, case["classes"], case["bf16"]))
    init = [gt[0]] + [T @ _random_pose(rng, 15.0, 0.05) for T in gt[1:]]
    return dict(xyz=xyz, sem=sem or None, rgb=None, edges=_all_pairs(K), poses=np.stack(init), ell=0.1,
                ell_color=0.0)


def _street_primitives(rng, half=8.0):
    x0, x1 = -70.0, 70.0
    boxes = [([x0, half, 0.0], [x1, half + 2.0, 15.0], 2), ([x0, -half - 2.0, 0.0], [x1, -half, 15.0], 3)]
    poles = []
    for side in (-1.0, 1.0):
        x = x0 + rng.uniform(0.0, 6.0)
        while x < x1 - 5.0:
            y, L, W, H = side * (half - 2.2), rng.uniform(3.8, 4.8), rng.uniform(1.7, 1.95), rng.uniform(1.4, 1.7)
            boxes.append(([x, y - W / 2, 0.0], [x + L, y + W / 2, H], 4 + int(rng.integers(0, 3))))
            x += L + rng.uniform(1.0, 9.0)
        x = x0 + rng.uniform(0.0, 10.0)
        while x < x1:
            poles.append((x, side * (half - 0.8), 0.12, 6.0, 7 + int(rng.integers(0, 2))))
            x += rng.uniform(8.0, 16.0)
    return boxes, poles


def _scan(g, T, boxes, poles, n_rays):
    """One 64-beam scan: frame-local points and their classes."""
    dd = dict(device=DEV, dtype=torch.float64)
    n_az = max(8, int(round(n_rays / 64)))
    el = torch.deg2rad(torch.linspace(-25.0, 3.0, 64, **dd))
    az = 2 * math.pi / n_az * (torch.arange(n_az, **dd) + float(_rand(g, 1)))
    E, A = torch.meshgrid(el, az, indexing="ij")
    local = torch.stack([torch.cos(E) * torch.cos(A), torch.cos(E) * torch.sin(A), torch.sin(E)], -1).reshape(-1, 3)
    local = torch.cat([local, local[:max(0, n_rays - len(local))]])[:n_rays]
    o = T[:3, 3]
    dirs = local @ torch.tensor(T[:3, :3].T.copy(), **dd)
    best = torch.full((n_rays,), math.inf, **dd)
    cls = torch.zeros(n_rays, device=DEV, dtype=torch.long)

    def hit(t, ok, c):
        ok = ok & (t > 0) & (t < best)
        best[:] = torch.where(ok, t, best)
        cls[:] = torch.where(ok, torch.full_like(cls, c), cls)

    hit(-o[2] / dirs[:, 2], dirs[:, 2] < 0, 0)
    for lo, hi, c in boxes:
        lo, hi = np.asarray(lo), np.asarray(hi)
        if np.linalg.norm(np.maximum(np.maximum(lo - o, o - hi), 0.0)) > 50.0:
            continue
        t1 = torch.tensor(lo - o, **dd) / dirs
        t2 = torch.tensor(hi - o, **dd) / dirs
        tmin = torch.minimum(t1, t2).amax(1)
        hit(tmin, torch.maximum(t1, t2).amin(1) >= tmin, c)
    for px, py, r, h, c in poles:
        dx, dy = o[0] - px, o[1] - py
        if math.hypot(dx, dy) - r > 50.0:
            continue
        a = dirs[:, 0] ** 2 + dirs[:, 1] ** 2
        b = 2 * (dx * dirs[:, 0] + dy * dirs[:, 1])
        disc = b * b - 4 * a * (dx * dx + dy * dy - r * r)
        t = (-b - disc.clamp(min=0).sqrt()) / (2 * a)
        z = o[2] + t * dirs[:, 2]
        hit(t, (disc > 0) & (z >= 0) & (z <= h), c)
    return local, best, cls


def _street_scene(case, seed, loop=False):
    g, rng = _gen(seed), np.random.default_rng(seed)
    K, n = case["frames"], case["points"]
    boxes, poles = _street_primitives(rng)
    window = case["op"] == "step"
    gt = []
    yaw, x, y = 0.0, -K / 2.0, 0.0
    for k in range(K):
        if loop:
            th = 2 * math.pi * k / 16
            gt.append(_pose(_rotation([0, 0, 1], th + math.pi / 2),
                            [16 / (2 * math.pi) * math.cos(th), 16 / (2 * math.pi) * math.sin(th), 1.7]))
        elif window:                        # a smooth path, 1 m between frames
            gt.append(_pose(_rotation([0, 0, 1], yaw), [x, y, 1.7]))
            yaw += math.radians(rng.normal(0.0, 1.5))
            x, y = x + math.cos(yaw), y + math.sin(yaw)
        else:
            gt.append(_pose(_rotation([0, 0, 1], math.radians(rng.uniform(-5, 5))),
                            [1.5 * k - 0.75 * (K - 1), rng.uniform(-1, 1), 1.7]))
    xyz, sem = [], []
    for T in gt:
        local, dist, cls = _scan(g, T, boxes, poles, n)
        keep = (dist >= 1.0) & (dist <= 50.0)
        dist = dist + (0.01 if not (loop or window) else 0.02) * _randn(g, n)
        pts, cls = (local * dist[:, None])[keep], cls[keep]
        if window:                          # a tenth of the points are outliers
            out = _rand(g, len(pts)) < 0.1
            lo, hi = pts.amin(0), pts.amax(0)
            pts = torch.where(out[:, None], lo + (hi - lo) * _rand(g, len(pts), 3), pts)
            cls = torch.where(out, (19 * _rand(g, len(pts))).long(), cls)
        xyz.append(pts.float().double())
        sem.append(_labels(g, cls, case["classes"], case["bf16"]))
    deg, trans = (1.0, 0.05) if loop else (2.0, 0.1) if window else (15.0, 0.5)
    if case["op"] in ("solve", "serve"):    # a front end's guess
        deg, trans = 2.0, 0.15
    edges = _all_pairs(K)
    if loop:
        edges = [(a, b) for a, b in edges
                 if b - a <= 7 or np.linalg.norm(gt[a][:3, 3] - gt[b][:3, 3]) < 0.5]
    init = [gt[0]] + [T @ _random_pose(rng, deg, trans) for T in gt[1:]]
    return dict(xyz=xyz, sem=sem, rgb=None, edges=edges, poses=np.stack(init), ell=0.3, ell_color=0.0)


def _scene(case, seed):
    if case["scene"] == "rgbd":
        s = _rgbd_scene(case, seed)
    elif case["scene"] == "object":
        s = _object_scene(case, seed)
    else:
        s = _street_scene(case, seed, case["scene"] == "loop")
    s["sizes"] = [len(x) for x in s["xyz"]]
    return s


def _requests(case, seed):
    """The served problems: frames and points spread over the case's range."""
    lo, hi, R = min(5000, case["points"]), case["points"], case["requests"]
    out = []
    for r in range(R):
        k = 2 + r % (case["frames"] - 1)
        n = int(round(lo * (hi / lo) ** ((r * 5 % R) / max(1, R - 1))))
        out.append(_scene(dict(case, frames=k, points=n), seed * 64 + 1 + r))
    return out


# ----------------------------------------------------------------- prepare --
def _params(case, s):
    return api.make_params(s["ell"], ell_color=s["ell_color"], sem_dim=case["classes"], sem_bf16=case["bf16"],
                           max_iters=case["iters"] or 100, top_k=case["top_k"], sem_min=case["sem_min"])


class _Resident:
    """A problem on the GPU: its inputs, and the library's context over them."""

    def __init__(self, case, seed, context=True):
        s = _scene(case, seed)
        self.K, self.E = len(s["sizes"]), len(s["edges"])
        self.sizes, self.edges, self.poses = s["sizes"], s["edges"], s["poses"]
        self.params = _params(case, s)
        self.xyz = torch.cat(s["xyz"]).contiguous()
        self.sem = torch.cat(s["sem"]).contiguous() if s["sem"] else None
        self.rgb = torch.cat(s["rgb"]).contiguous() if s["rgb"] else None
        self.d_poses = torch.tensor(self.poses, device=DEV).contiguous()
        torch.cuda.synchronize()             # the library runs on its own stream
        self.ctx = self.create() if context else None
        if context and case["unit_queries"] != 32:
            api.rkhsba_set_tuning(self.ctx, case["unit_queries"], 0)

    def pointers(self):
        return [None if t is None else t.data_ptr() for t in (self.xyz, self.sem, self.rgb)]

    def create(self):
        return api.rkhsba_create_device(self.sizes, *self.pointers(), self.edges, self.params)

    def __del__(self):
        if getattr(self, "ctx", None):
            api.rkhsba_destroy(self.ctx)
            self.ctx = None


class _Serving:
    """A running server and the requests in hand, as host arrays."""

    def __init__(self, case, seed):
        self.server = pk.Server(max_inflight=8)
        self.probs = []
        for s in _requests(case, seed):
            self.probs.append(dict(xyz=[x.cpu().numpy() for x in s["xyz"]], sem=[x.cpu().numpy() for x in s["sem"]],
                                   edges=np.asarray(s["edges"], np.int32), poses0=s["poses"],
                                   params=dict(ell=s["ell"], sem_bf16=int(case["bf16"]), max_iters=case["iters"])))

    def __del__(self):
        if getattr(self, "server", None):
            self.server.close()
            self.server = None


def prepare(case, seed):
    if case["op"] == "serve":
        return dict(op="serve", s=_Serving(case, seed))
    return dict(op=case["op"], iters=case["iters"], s=_Resident(case, seed, case["op"] not in ("static", "fresh")))


# --------------------------------------------------------------------- run --
def _f32(x):
    return np.asarray(x).astype(np.float32)


def _evaluation(r):
    return dict(loss=_f32(r["loss"]), grad=_f32(r["grad"]), H=_f32(r["H"]), pairs=r["edge_pairs"])


def _solution(T, info):
    return dict(poses=_f32(T), loss=_f32(info["final_loss"]), iters=info["iters"])


def run(state):
    op, s = state["op"], state["s"]
    if op == "eval":
        return _evaluation(api.rkhsba_eval(s.ctx, s.poses, s.K, s.E))
    if op == "static":
        r = api.rkhsba_eval_static(s.sizes, *s.pointers(), s.edges, s.params, s.poses)
        return dict(loss=_f32(r["loss"]), grad=_f32(r["grad"]), H=_f32(r["H"]))
    if op == "solve":
        return _solution(*api.rkhsba_solve(s.ctx, s.poses, s.K))
    if op == "step":
        api.rkhsba_rebuild(s.ctx)
        api.rkhsba_set_poses_device(s.ctx, s.d_poses.data_ptr())
        api.rkhsba_iterate(s.ctx, state["iters"])
        return _solution(*api.rkhsba_get_state(s.ctx, s.K))
    if op == "fresh":
        ctx = s.create()
        r = api.rkhsba_eval(ctx, s.poses, s.K, s.E)
        api.rkhsba_destroy(ctx)
        return _evaluation(r)
    if op == "search":
        r = api.rkhsba_rotation_search(s.ctx, 0, 1, s.poses, s.K)
        return dict(cos=_f32(r["cos"]), best=r["best"], pose=_f32(r["best_pose"]))
    if op == "distance":
        r = api.rkhsba_inner_products(s.ctx, s.poses, s.K, s.E)
        return {k: _f32(v) for k, v in r.items()}
    tickets = [s.server.submit(p) for p in s.probs]
    done = [s.server.poll(t) for t in tickets]
    return [_solution(T, i) for T, i in done]


# -------------------------------------------------------------------- work --
def _neighbours(case):
    """Pairs inside the cutoff per point and edge, about (counted on these scenes)."""
    n = case["points"]
    return n * {"rgbd": 0.0004, "object": 0.23, "street": 0.0045, "loop": 0.0082}[case["scene"]]


def _pairs(case):
    """Pair-terms of one pass, about."""
    if case["op"] == "serve":
        K, n = 0.5 * (2 + case["frames"]), math.sqrt(min(5000, case["points"]) * case["points"])
        times = case["requests"] * (1 + case["iters"])
    else:
        K, n = case["frames"], case["points"]
        times = {"solve": 1 + case["iters"], "step": 1 + case["iters"], "search": 60}.get(case["op"], 1)
    edges = K * (K - 1) / 2
    if case["scene"] == "loop":
        k = case["frames"]
        edges = sum(1 for a in range(k) for b in range(a + 1, k) if b - a <= 7 or (b - a) % 16 == 0)
    return edges * n * _neighbours(dict(case, points=n)) * times


def work(case):
    K, n, label = case["frames"], case["points"], 2 if case["bf16"] else 4
    if case["op"] == "serve":
        K, n = 0.5 * (2 + K) * case["requests"], math.sqrt(min(5000, n) * n)
    read = K * n * (24 + label * case["classes"] + (12 if case["colour"] else 0))
    return {"bytes": read + 8.0 * (6 * K) ** 2, "flops": _pairs(case) * (72 + 2 * case["classes"])}


# ------------------------------------------------------------------- exact --
# The paper's sums in 64 bits with plain torch: for every edge (a, b) the points
# of b are moved into frame a, taken in blocks of near points, and paired with
# the points of a around the block.
def _near_blocks(y, size, block=1024):
    cell = torch.floor(y / size).long()
    cell = (cell - cell.amin(0)).clamp_(max=1023)
    key = torch.zeros_like(cell[:, 0])
    for bit in range(10):                     # cells along a Morton curve
        for k in range(3):
            key |= ((cell[:, k] >> bit) & 1) << (3 * bit + k)
    return torch.argsort(key, stable=True).split(block)


def _edge_sums(case, s, a, b, Ta, Tb):
    """sum w, w d, w x d^T, ... of one edge in world axes: (F, E2, grad 12, H 12x12)."""
    dd = dict(device=DEV, dtype=torch.float64)
    rc, kg = 3.0 * s["ell"], -0.5 / s["ell"] ** 2
    Ra, ta, Rb, tb = (torch.tensor(v, **dd) for v in (Ta[:3, :3], Ta[:3, 3], Tb[:3, :3], Tb[:3, 3]))
    xa, xb = s["xyz"][a], s["xyz"][b]
    out = torch.zeros(1 + 1 + 12 + 144, **dd)
    if not len(xa) or not len(xb):
        return out
    X, Y = xa @ Ra.T + ta, xb @ Rb.T + tb
    centre = X.mean(0)
    total = torch.zeros(10, 10, **dd)         # sum w phi(x) phi(y)^T, phi = (1, z, z z^T), z about the centre
    E2 = torch.zeros((), **dd)

    def phi(p):
        p = p - centre
        return torch.cat([torch.ones_like(p[:, :1]), p, p[:, :1] * p, p[:, 1:2] * p[:, 1:], p[:, 2:] * p[:, 2:]], 1)

    FX, FY = phi(X), phi(Y)
    for idx in _near_blocks(Y, rc):
        q = Y[idx]
        lo, hi = q.amin(0) - rc, q.amax(0) + rc
        near = ((X >= lo) & (X <= hi)).all(1).nonzero()[:, 0]
        for c in near.split(32768):
            x = X[c]
            r2 = torch.zeros(len(idx), len(c), **dd)
            for k in range(3):
                r2.add_((q[:, k:k + 1] - x[None, :, k]).square_())
            w = torch.exp(kg * r2)
            if case["colour"] and s["rgb"] is not None and s["ell_color"] > 0:
                cr, cq = s["rgb"][a][c].double(), s["rgb"][b][idx].double()
                for k in range(3):
                    w.mul_(torch.exp(-0.5 / s["ell_color"] ** 2 * (cq[:, k:k + 1] - cr[None, :, k]).square_()))
            if s["sem"]:
                lab = s["sem"][b][idx].double() @ s["sem"][a][c].double().T
                if case["sem_min"] > 0:
                    w.mul_(lab >= case["sem_min"])
                w.mul_(lab)
            w.mul_(r2 < rc * rc)
            if case["top_k"]:
                # all candidates of a query are in one split here (top_k cases are small)
                kth = torch.topk(w, min(case["top_k"], w.shape[1]), 1).values[:, -1:]
                w = torch.where(w >= kth, w, torch.zeros_like(w))
            total += FX[c].T @ (w.T @ FY[idx])
            E2 += (w * r2).sum()
    # moments of z = x - centre, u = y - centre in world axes
    W, sx, sy = total[0, 0], total[1:4, 0], total[0, 1:4]
    up = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
    Mxx, Myy, Mxy = torch.zeros(3, 3, **dd), torch.zeros(3, 3, **dd), total[1:4, 1:4]
    for t, (i, j) in enumerate(up):
        Mxx[i, j] = Mxx[j, i] = total[4 + t, 0]
        Myy[i, j] = Myy[j, i] = total[0, 4 + t]
    # body-frame quantities: p = R^T (x_world - t), d = x_world - y_world
    ca, cb = Ra.T @ (centre - ta), Rb.T @ (centre - tb)
    D = sx - sy
    Kx = Mxx - Mxy                            # sum w z d^T
    Ky = Mxy.T - Myy                          # sum w u d^T
    A = Ra.T @ Kx @ Ra + torch.outer(ca, Ra.T @ D)        # sum w p_a (R_a^T d)^T
    B = Rb.T @ Ky @ Rb + torch.outer(cb, Rb.T @ D)

    def axial(M):                             # sum p x d from sum p d^T
        return torch.stack([M[1, 2] - M[2, 1], M[2, 0] - M[0, 2], M[0, 1] - M[1, 0]])

    def skew(v):
        S = torch.zeros(3, 3, **dd)
        S[0, 1], S[0, 2], S[1, 2] = -v[2], v[1], -v[0]
        return S - S.T

    grad = torch.cat([Ra.T @ D, axial(A), -(Rb.T @ D), -axial(B)])
    Pa, Pb = Ra.T @ sx + W * ca, Rb.T @ sy + W * cb       # sum w p
    za, zb = Ra.T @ sx, Rb.T @ sy
    Qa = Ra.T @ Mxx @ Ra + torch.outer(za, ca) + torch.outer(ca, za) + W * torch.outer(ca, ca)
    Qb = Rb.T @ Myy @ Rb + torch.outer(zb, cb) + torch.outer(cb, zb) + W * torch.outer(cb, cb)
    Qab = Ra.T @ Mxy @ Rb + torch.outer(za, cb) + torch.outer(ca, zb) + W * torch.outer(ca, cb)
    R = Ra.T @ Rb                             # J_a = R_a [I, -[p]x], J_b = -R_b [I, -[q]x]
    I3 = torch.eye(3, **dd)
    H = torch.zeros(12, 12, **dd)
    for o, P, Q in ((0, Pa, Qa), (6, Pb, Qb)):
        H[o:o + 3, o:o + 3] = W * I3
        H[o:o + 3, o + 3:o + 6] = -skew(P)
        H[o + 3:o + 6, o:o + 3] = skew(P)
        H[o + 3:o + 6, o + 3:o + 6] = Q.trace() * I3 - Q
    basis = [skew(I3[k]) for k in range(3)]
    G = torch.zeros(3, 3, **dd)               # sum w [p]x^T R [q]x
    for i in range(3):
        for j in range(3):
            G += Qab[i, j] * (basis[i].T @ R @ basis[j])
    H[0:3, 6:9] = -W * R
    H[0:3, 9:12] = R @ skew(Pb)
    H[3:6, 6:9] = skew(Pa).T @ R
    H[3:6, 9:12] = -G
    H[6:12, 0:6] = H[0:6, 6:12].T
    return torch.cat([W[None], E2[None], grad, H.reshape(-1)])


def _system(case, s, poses):
    K = len(s["sizes"])
    F, grad, H, per = 0.0, np.zeros(6 * K), np.zeros((6 * K, 6 * K)), []
    for a, b in s["edges"]:
        v = _edge_sums(case, s, a, b, poses[a], poses[b]).cpu().numpy()
        ix = np.r_[6 * a:6 * a + 6, 6 * b:6 * b + 6]
        F += v[0]
        grad[ix] += v[2:14]
        H[np.ix_(ix, ix)] += v[14:].reshape(12, 12)
        per.append((v[0], v[1]))
    return F, grad, H, per


def _exp(xi):
    rho, th = xi[:3], np.linalg.norm(xi[3:])
    P = np.array([[0, -xi[5], xi[4]], [xi[5], 0, -xi[3]], [-xi[4], xi[3], 0]])
    if th < 1e-5:
        A, B, C = 1 - th * th / 6, 0.5 - th * th / 24, 1 / 6 - th * th / 120
    else:
        A, B, C = math.sin(th) / th, (1 - math.cos(th)) / th ** 2, (th - math.sin(th)) / th ** 3
    return _pose(np.eye(3) + A * P + B * P @ P, (np.eye(3) + B * P + C * P @ P) @ rho)


def _levenberg_marquardt(case, s, iters):
    T, lam = s["poses"].copy(), 1e-4
    F, b, H, _ = _system(case, s, T)
    done = 0
    for _ in range(iters):
        Hf, bf = H[6:, 6:], b[6:]
        dm = np.diag(Hf)
        A = Hf + lam * np.diag(np.maximum(dm, 1e-9 * dm.max()))
        delta = np.linalg.solve(A, -bf)
        Tn = T.copy()
        for m in range(1, len(T)):
            Tn[m] = T[m] @ _exp(delta[6 * (m - 1):6 * m])
        Fn, bn, Hn, _ = _system(case, s, Tn)
        done += 1
        step = np.abs(delta).max()
        if Fn > F:
            rel = (Fn - F) / max(abs(F), 1e-300)
            T, F, b, H, lam = Tn, Fn, bn, Hn, max(0.1 * lam, 1e-12)
            if step < 1e-10 or rel < 1e-12:
                break
        else:
            lam *= 10
            if step < 1e-10 or lam > 1e10:
                break
    return dict(poses=T, loss=np.float64(-F), iters=None)


def _self_terms(case, s, m):
    eye = np.eye(4)
    v = _edge_sums(case, dict(s, sizes=s["sizes"]), m, m, eye, eye)
    return float(v[0]), float(v[1])


def _rotations():
    phi = (1 + math.sqrt(5)) / 2
    gens = [_rotation([0.0, 1.0, phi], 2 * math.pi / 5), _rotation([0.0, 0.0, 1.0], math.pi)]
    group, i = [np.eye(3)], 0
    while i < len(group):
        for g in gens:
            P = group[i] @ g
            if not any(np.abs(P - Q).max() < 1e-9 for Q in group):
                group.append(P)
        i += 1
    # half turns, third turns, fifth turns by the trace; by the entries inside a class
    order = lambda A: ([3, -1, 0].index(round(np.trace(A), 6)) if round(np.trace(A), 6) in (3, -1, 0) else 3,
                       tuple(np.round(A, 7).ravel() + 0.0))
    return sorted(group, key=order)


def exact(case, seed):
    if case["op"] == "serve":
        return [_levenberg_marquardt(case, s, case["iters"]) for s in _requests(case, seed)]
    if _pairs(case) > 1.2e10:
        return None                           # tens of billions of pairs: over 20 seconds in 64 bits
    s = _scene(case, seed)
    if case["op"] in ("solve", "step"):
        return _levenberg_marquardt(case, s, case["iters"])
    if case["op"] == "search":
        mu = [x.mean(0).cpu().numpy() for x in s["xyz"]]
        norm = math.sqrt(_self_terms(case, s, 0)[0] * _self_terms(case, s, 1)[0])
        cos, poses = [], []
        for Q in _rotations():
            P = s["poses"][0] @ _pose(Q, mu[0] - Q @ mu[1])
            cos.append(float(_edge_sums(case, s, 0, 1, s["poses"][0], P)[0]) / norm)
            poses.append(P)
        return dict(cos=np.array(cos), best=None, pose=poses[int(np.argmax(cos))])
    F, grad, H, per = _system(case, s, s["poses"])
    if case["op"] == "distance":
        self_terms = [_self_terms(case, s, m) for m in range(len(s["sizes"]))]
        S, X = np.array([v[0] for v in self_terms]), np.array([v[0] for v in per])
        e = np.asarray(s["edges"])
        E2 = sum(self_terms[a][1] + self_terms[b][1] - 2 * p[1] for (a, b), p in zip(s["edges"], per))
        return {"self": S, "cross": X, "dist": S[e[:, 0]] + S[e[:, 1]] - 2 * X,
                "cos": X / np.sqrt(S[e[:, 0]] * S[e[:, 1]]), "dD_dell": np.float64(E2 / s["ell"] ** 3)}
    out = dict(loss=np.float64(-F), grad=grad / s["ell"] ** 2, H=H)
    return out if case["op"] == "static" else dict(out, pairs=None)

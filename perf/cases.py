"""The work whose time is measured: calls of the library's public entry points
(paper_2302_11815_gb300.wost) as a user's program makes them.

A case names a scene of scenes.py, an entry point ("call") and its sizes:

  solve    wost.solve: create, wait, poll, destroy, from host or device points
  static   wost_solve_static: the solve that allocates nothing
  batch    wost_solve_batch over several scenes
  engine   a few requests through the serving engine, until all are answered
  queries  Q.1-Q.4 over arrays of queries

The scenes stay what they are (a user's geometry is given once and kept
resident); the evaluation points, the queries and the walks' random key come
from the seed.  The walks are single precision and their estimates carry a
sampling error of a percent or more, so the solution is kept as a float32
field, as the static solve writes it.  Every output of a call that is a
result is returned (mean, standard error, walks per point; distance, closest
point, primitive, ...); its progress record (clock times) is not one.
"""
import functools
import math

import numpy as np
import torch

from paper_2302_11815_gb300 import scenes, wost


def listed():
    return [
        # A probe of a few points on a small double-sided domain (a crack, App. B) from host arrays, the
        # one-launch kernel: the call is launches, copies and allocations.
        dict(name="probe_crack", call="solve", scene="crack", size=16, points=24, walks=32, kernel="plain",
             host=True),
        # The README's example: the 64-gon flower, half Neumann, 256 points, 512 walks.
        dict(name="flower", call="solve", scene="flower", size=64, points=256, walks=512, kernel="persistent",
             host=False),
        # Neumann-dominated rooms: walks of some hundred steps, few of them, the regime of long tails.
        dict(name="keyhole", call="solve", scene="keyhole", size=20, points=64, walks=96, kernel="persistent",
             host=False),
        # The lung-like field of the headline workload, a preview: few walks at scattered raster points, whose
        # longest walk is all that is left to wait for.
        dict(name="koch_preview", call="solve", scene="koch", size=5, points=61, walks=16, kernel="persistent",
             host=False, cap=65536),
        # The same field solved in earnest, by the resumable form that long solves use, from host points, under the
        # step cap of the batched workload.
        dict(name="koch_field", call="solve", scene="koch", size=5, points=997, walks=128, kernel="resumable",
             host=True, cap=16384),
        # A screened problem (reaction-diffusion) on a disk, half Neumann.
        dict(name="screened_disk", call="solve", scene="disk", size=128, points=1001, walks=256,
             kernel="persistent", host=False, sigma=1.93),
        # 3D: a raster of a slice plane around the noisy torus (200,000 Neumann triangles), few walks per point.
        dict(name="torus_slice", call="solve", scene="torus", size=500, points=17003, walks=32,
             kernel="persistent", host=False),
        # 3D, a small mesh and many points in the form without allocation (an update per frame).
        dict(name="static_box", call="static", scene="box_sphere", size=6, points=65000, walks=4),
        # A mixture of 2D and 3D problems of uneven size in one batched launch.
        dict(name="batch_mix", call="batch", scenes=12, prims=20000, points=400, walks=64),
        # Requests to the serving engine: two resident scenes, an accuracy target each.
        dict(name="engine_mix", call="engine", requests=6, points=700, walks=256, target=0.03),
        # The geometric queries by themselves: a handful in 2D, and a slice raster in 3D.
        dict(name="queries_koch", call="queries", scene="koch", size=5, points=1000),
        dict(name="queries_torus", call="queries", scene="torus", size=500, points=250007),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "solve", "static", "batch", "engine", "queries"])
    if call == "batch":
        return dict(call=call, scenes=rng.randint(2, 16), prims=_logint(rng, 1000, 30000),
                    points=_logint(rng, 5, 500), walks=_logint(rng, 16, 64))
    if call == "engine":
        return dict(call=call, requests=rng.randint(1, 8), points=_logint(rng, 50, 1000),
                    walks=_logint(rng, 64, 256), target=round(rng.uniform(0.02, 0.08), 4))
    scene = rng.choice(["crack", "flower", "keyhole", "koch", "disk", "torus", "box_sphere", "annulus"])
    size = {"crack": rng.randint(8, 40), "flower": 64, "keyhole": rng.randint(10, 40), "koch": rng.randint(2, 5),
            "disk": _logint(rng, 32, 700), "torus": rng.choice([60, 125, 250, 500]), "box_sphere": rng.randint(2, 10),
            "annulus": _logint(rng, 24, 500)}[scene]
    if call == "queries":
        return dict(call=call, scene=scene, size=size, points=_logint(rng, 100, 250000))
    # walks of one call: what the longest listed case of the scene's kind runs, at most
    most = {"keyhole": 20000, "koch": 150000}.get(scene, 500000)
    walks = _logint(rng, 4, 512)
    points = _logint(rng, 8, max(9, min(60000, most // walks)))
    if call == "static":
        return dict(call=call, scene=scene, size=size, points=points, walks=walks)
    case = dict(call=call, scene=scene, size=size, points=points, walks=walks,
                kernel=rng.choice(["plain", "persistent", "persistent", "resumable"]), host=rng.random() < 0.4)
    if scene in ("disk", "annulus") and rng.random() < 0.5:
        case["sigma"] = round(math.exp(rng.uniform(math.log(0.05), math.log(50.0))), 4)
    if scene in ("keyhole", "koch") and case["kernel"] == "plain":
        case["kernel"] = "resumable"
    if scene == "koch":
        case["cap"] = rng.choice([1024, 8192, 16384])
    return case


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
_DISK_A = (1.2, -0.7)  # u = exp(a.x) solves the screened equation with sigma = |a|^2 = 1.93


@functools.lru_cache(maxsize=None)
def _spec(scene, size):
    """The scene's description: geometry and boundary data (never changed)."""
    if scene == "crack":
        return scenes.crack_square_scene(m=size, n_slit=size)
    if scene == "flower":
        return scenes.config1(n_points=1)
    if scene == "keyhole":
        return scenes.keyhole_scene(seg=1.0 / size, n_points=1)
    if scene == "koch":
        return scenes.config2(grid=8, level=size)
    if scene == "disk":
        return scenes.disk_scene(size, "exp_plane", (1.0, *_DISK_A, 0.0), neumann=np.arange(size) < size // 2)
    if scene == "torus":
        return scenes.config3(grid=4, nu=size, nv=max(8, 2 * size // 5))
    if scene == "box_sphere":
        return scenes.box_sphere_scene(m=size, n_lat=2 * size + 4, n_lon=4 * size + 8)
    if scene == "annulus":
        return scenes.annulus_scene(2 * size, size)
    raise ValueError(scene)


@functools.lru_cache(maxsize=None)
def _batch_specs(n, prims, points, walks):
    return scenes.config4(n_scenes=n, prims=(1e3, prims), points=(1, points), walks=(16, max(17, walks)))


# epsilon, r_min and the step cap of each scene: those of its configuration, or of its tests
_EPS = {"koch": 1e-4}
_CAP = {"flower": 1024, "torus": 1024, "koch": 8192, "keyhole": 1 << 20}

_resident = {}


def _scene(scene, size):
    """A scene's handle: the large 3D ones stay resident between requests, the others are set up anew."""
    if scene != "torus":
        return wost.Scene(_spec(scene, size))
    if (scene, size) not in _resident:
        _resident[scene, size] = wost.Scene(_spec(scene, size))
    return _resident[scene, size]


def _outline(scene, size):
    """Outer boundary and holes of a 2D scene as closed polygons."""
    V = _spec(scene, size)["vertices"].astype(np.float64)
    if scene == "koch":
        n = 3 * 4**size
        return V[:n], [V[n:]]
    return V, []


def _points(rng, scene, size, n):
    if scene == "crack":
        p = rng.uniform(-0.95, 0.95, (n, 2))
        p[:, 1] += np.where(p[:, 1] < 0, -0.02, 0.02)  # off the crack
    elif scene in ("flower", "koch"):
        outer, holes = _outline(scene, size)
        if scene == "koch":  # cell centres of the workload's 512 x 512 raster, scattered over the domain
            lo, hi = outer.min(0), outer.max(0)
            got, have = [], 0
            while have < n:
                c = lo + (rng.integers(0, 512, (2 * n + 16, 2)) + 0.5) / 512 * (hi - lo)
                ok = scenes._inside_chunked(c, outer) & ~scenes._inside_chunked(c, holes[0])
                got.append(c[ok])
                have += len(got[-1])
            p = np.concatenate(got)[:n]
        else:
            p = scenes.sample_inside_2d(rng, n, outer)
    elif scene == "keyhole":
        p = np.c_[rng.uniform(-1.9, -0.1, n), rng.uniform(-0.9, 0.9, n)]
    elif scene == "disk":
        p = scenes.ball_points(rng, n, 2, 0.85)
    elif scene == "annulus":
        r, t = np.sqrt(rng.uniform(0.35**2, 0.95**2, n)), rng.uniform(0, 2 * np.pi, n)
        p = np.c_[r * np.cos(t), r * np.sin(t)]
    elif scene == "box_sphere":
        p = rng.uniform(-0.95, 0.95, (2 * n + 64, 3))
        p = p[np.linalg.norm(p, axis=1) > 0.42][:n]
    else:  # torus: a raster of a plane through the cube, in raster order, outside the (noisy) tube
        axis, off = int(rng.integers(3)), rng.uniform(-0.9, 0.9)
        m = int(math.sqrt(1.3 * n)) + 4
        while True:
            s = (np.arange(m) + 0.5) / m * 2 - 1
            a, b = np.meshgrid(s, s, indexing="ij")
            p = np.insert(np.stack([a.ravel(), b.ravel()], 1), axis, off, axis=1)
            p = p[np.hypot(np.hypot(p[:, 0], p[:, 1]) - 0.5, p[:, 2]) > 0.235]
            if len(p) >= n:
                break
            m += max(1, m // 8)
        p = p[:n]
    return np.ascontiguousarray(p, np.float32)


class _State:
    """What a user's program holds; its engine ends before its scenes do."""

    engine = None

    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        if self.engine is not None:
            wost.wost_engine_destroy(self.engine)
            self.engine = None


# ---------------------------------------------------------------------------
# the measured calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    rng = np.random.default_rng(seed)
    key = int(rng.integers(1 << 62))
    call = case["call"]
    if call == "batch":
        specs = _batch_specs(case["scenes"], case["prims"], case["points"], case["walks"])
        pts = [torch.from_numpy(sc["points"][rng.permutation(len(sc["points"]))]).cuda() for sc in specs]
        return _State(call=call, scenes=[wost.Scene(sc) for sc in specs],
                      requests=[dict(points=p, walks_per_point=sc["walks"], epsilon=sc["epsilon"], r_min=sc["r_min"],
                                     max_steps=sc["max_steps"], seed=key + i) for i, (sc, p) in
                                enumerate(zip(specs, pts))])
    if call == "engine":
        held = [("flower", 64), ("box_sphere", 6)]
        handles = [wost.Scene(_spec(*h)) for h in held]
        reqs = []
        for i in range(case["requests"]):
            k = i % 2
            n = max(1, case["points"] // (1 + i % 3))
            reqs.append((handles[k].handle, _points(rng, *held[k], n), case["target"] * (1 + i % 2)))
        return _State(call=call, scenes=handles, requests=reqs, walks=case["walks"], key=key,
                      engine=wost.wost_engine_create())
    scene, size, n = case["scene"], case["size"], case["points"]
    S = _scene(scene, size)
    pts = _points(rng, scene, size, n)
    if call == "queries":
        dim = S.dim
        d = rng.normal(size=(n, dim))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
        return _State(call=call, scene=S, points=dev(pts), dirs=dev(d), reach=dev(rng.uniform(0.3, 1.0, n)),
                      radius=dev(rng.uniform(0.05, 0.6, n)), key=key)
    common = dict(walks=case["walks"], epsilon=_EPS.get(scene, 1e-3), r_min=_EPS.get(scene, 1e-3),
                  max_steps=case.get("cap", _CAP.get(scene, 4096)), seed=key)
    if call == "static":
        dev = torch.from_numpy(pts).cuda()
        return _State(call=call, scene=S, points=dev, common=common, mean=torch.empty(n, device="cuda"),
                      se=torch.empty(n, device="cuda"))
    return _State(call=call, scene=S, points=pts if case["host"] else torch.from_numpy(pts).cuda(), common=common,
                  more=dict(kernel=case["kernel"], sigma=case.get("sigma", 0.0)))


def _field(mean, se, walks):
    return {"mean": mean.astype(np.float32), "se": se.astype(np.float32), "walks": walks.astype(np.int64)}


def run(state):
    s = state
    if s.call == "solve":
        r = wost.solve(s.scene, s.points, **s.common, **s.more)
        return _field(r["mean"], r["se"], r["walks"])
    if s.call == "static":
        c = s.common
        wost.wost_solve_static(s.scene.handle, s.points, c["walks"], c["epsilon"], c["r_min"], c["max_steps"],
                               c["seed"], 0, s.mean, s.se)
        return {"mean": s.mean, "se": s.se}
    if s.call == "batch":
        handles = wost.wost_solve_batch([S.handle for S in s.scenes], s.requests)
        out = []
        for h, q in zip(handles, s.requests):
            wost.wost_wait(h)
            out.append(_field(*wost.wost_poll(h, q["points"].shape[0])[:3]))
            wost.wost_solve_destroy(h)
        return out
    if s.call == "engine":
        handles = [wost.wost_engine_submit(s.engine, scene, pts, target, s.walks, 1e-3, 1e-3, 4096, seed=s.key + i)
                   for i, (scene, pts, target) in enumerate(s.requests)]
        out = []
        for h, (_, pts, _) in zip(handles, s.requests):
            wost.wost_wait(h)
            out.append(_field(*wost.wost_poll(h, len(pts))[:3]))
            wost.wost_solve_destroy(h)
        return out
    scene = s.scene.handle
    dist, closest, prim = wost.wost_query_closest_dirichlet(scene, s.points)
    sil = wost.wost_query_silhouette(scene, s.points, s.radius)
    hit, t, hprim = wost.wost_query_intersect_neumann(scene, s.points, s.dirs, s.reach)
    z, pdf, zprim = wost.wost_query_neumann_sample(scene, s.points, s.radius, s.key, 1, 2)
    return {"dist": dist, "closest": closest, "prim": prim, "sil": sil, "hit": hit, "t": t, "hprim": hprim, "z": z,
            "pdf": pdf, "zprim": zprim}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# Mean steps of a walk, and the least arithmetic of a step: each tree is gone down once (Q.1, Q.2, Q.3 visit a node
# per level, two box tests each) and a leaf of about two primitives tested; some 60 operations for the step itself.
_STEPS = {"crack": 20, "flower": 16, "keyhole": 330, "koch": 3000, "disk": 14, "torus": 40, "box_sphere": 23,
          "annulus": 24}


def _step_flops(prims, dim):
    levels = max(1.0, math.log2(max(2, prims) / 2))
    return 3 * levels * 2 * (8 if dim == 2 else 12) + 6 * (20 if dim == 2 else 60) + 60


def _walk_work(points, walks, steps, prims, dim):
    scene_bytes = prims * (16 * 3 if dim == 2 else 48 * 3)
    return {"bytes": scene_bytes + points * (4 * dim + 16), "flops": points * walks * steps * _step_flops(prims, dim)}


def work(case):
    call = case["call"]
    if call == "batch":
        w = [_walk_work(len(sc["points"]), sc["walks"], 60, len(sc["prims"]), sc["dim"])
             for sc in _batch_specs(case["scenes"], case["prims"], case["points"], case["walks"])]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if call == "engine":  # at least the first stage's walks of every request
        w = [_walk_work(max(1, case["points"] // (1 + i % 3)), 16, 12, 64 if i % 2 == 0 else 1392, 2 + i % 2)
             for i in range(case["requests"])]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    sc = _spec(case["scene"], case["size"])
    dim, prims, n = sc["dim"], len(sc["prims"]), case["points"]
    if call == "queries":  # points, directions, reaches in; three distances, three ids, two points, pdf, hit out
        return {"bytes": prims * (16 * 3 if dim == 2 else 48 * 3) + n * 4 * (4 * dim + 2 + 8),
                "flops": n * (4 / 3) * _step_flops(prims, dim)}
    return _walk_work(n, case["walks"], _STEPS[case["scene"]], prims, dim)


# ---------------------------------------------------------------------------
# values in 64 bits
# ---------------------------------------------------------------------------
def _u(scene, x):
    """The solution of the problem: what the walks' mean estimates."""
    x = x.astype(np.float64)
    if scene == "flower":
        return np.exp(x[:, 0]) * np.cos(x[:, 1])
    if scene == "disk":
        return np.exp(x @ np.array(_DISK_A))
    if scene == "box_sphere":
        return x[:, 0] ** 2 - x[:, 1] ** 2 + 0.5 * x[:, 2]
    if scene == "annulus":
        return 1.0 + 0.5 * np.log(np.hypot(x[:, 0], x[:, 1]))
    return None


def _segments_closest(V, x):
    """Distance and closest point of x to the segments V [m, 2, 2], in 64 bits, by all pairs."""
    a, e = V[:, 0], V[:, 1] - V[:, 0]
    dist = torch.full((len(x),), math.inf, dtype=torch.float64, device=x.device)
    point = torch.zeros_like(x)
    for i in range(0, len(x), 4096):
        q = x[i:i + 4096, None, :]
        t = (((q - a) * e).sum(-1) / (e * e).sum(-1)).clamp(0, 1)
        c = a + t[..., None] * e
        d, k = ((q - c) ** 2).sum(-1).min(1)
        dist[i:i + 4096] = d.sqrt()
        point[i:i + 4096] = c[torch.arange(len(k), device=x.device), k]
    return dist, point


def _box_faces_closest(x):
    """Distance from points inside the cube [-1, 1]^3 to its faces, and the closest point, in 64 bits."""
    d, axis = (1 - x.abs()).min(1)
    point = x.clone()
    row = torch.arange(len(x), device=x.device)
    point[row, axis] = torch.sign(x[row, axis])
    return d, point


def exact(case, seed):
    """The problem's solution for the mean of a solve with enough walks that the sampling error is small beside it
    (the sampled estimate itself has no 64-bit value: it is a random variable of the walks' single-precision
    paths); the distances and closest points of Q.1, whose value is plain geometry."""
    rng = np.random.default_rng(seed)
    rng.integers(1 << 62)
    call = case["call"]
    if call == "solve" and case["walks"] >= 256 and (case["scene"] == "disk") == ("sigma" in case):
        if "sigma" in case and abs(case["sigma"] - 1.93) > 1e-9:
            return None
        u = _u(case["scene"], _points(rng, case["scene"], case["size"], case["points"]))
        return None if u is None else {"mean": u, "se": None, "walks": None}
    if call == "queries":
        sc = _spec(case["scene"], case["size"])
        x = torch.from_numpy(_points(rng, case["scene"], case["size"], case["points"])).cuda().double()
        if sc["dim"] == 2:
            on = sc["prims"][(sc["flags"] & 1) == 0]
            if len(on) * len(x) > 1 << 30:
                return None
            dist, closest = _segments_closest(torch.from_numpy(sc["vertices"][on]).cuda().double(), x)
        else:  # the Dirichlet part of both 3D scenes is the cube
            dist, closest = _box_faces_closest(x)
        return {"dist": dist, "closest": closest}
    return None

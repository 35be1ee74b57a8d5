"""Walks carried by whole warps (small solves, and the last walks of large
ones) are those of the one-lane kernels, bit for bit: same step counts, means
that differ by the order of the FP64 additions only (1e-9, as between the
one-lane kernels).  A solve that gives its traversal limits itself (here: the
scene's own) stays on the one-lane kernels, which are tested against the
oracle."""
import numpy as np
import pytest

from paper_2302_11815_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wost():
    from paper_2302_11815_gb300 import build as libbuild
    from paper_2302_11815_gb300 import wost as w

    assert torch.cuda.is_available()
    libbuild.build()
    w.load()
    return w


def _disk(frac):
    n = 300
    return scenes.disk_scene(n, "exp_plane", (1.0, 1.2, -0.7, 0.0), neumann=np.arange(n) < frac * n)


def _moved(sc, shift):
    """The scene away from the origin: the rounding of positions grows with them."""
    sc = dict(sc)
    sc["vertices"] = (sc["vertices"] + np.float32(shift)).astype(np.float32)
    return sc


CASES = {
    "flower": (lambda: scenes.config1(), 0, 0.0),
    "flower_leaf16": (lambda: scenes.config1(data="per_vertex"), 16, 0.0),
    "flower_far": (lambda: _moved(scenes.config1(), 30.0), 0, 0.0),
    "koch3": (lambda: scenes.config2(grid=8, level=3), 0, 0.0),
    "koch4_leaf1": (lambda: scenes.config2(grid=8, level=4), 1, 0.0),
    "keyhole": (lambda: scenes.keyhole_scene(), 0, 0.0),
    "square": (lambda: scenes.square_scene(200, neumann_sides=("left", "bottom")), 0, 0.0),
    "crack": (lambda: scenes.crack_square_scene(), 0, 0.0),
    "slit": (lambda: scenes.slit_square_scene(), 2, 0.0),
    "sheet": (lambda: scenes.sheet_square_scene(m=60, n_sheet=90, data="per_corner_minus"), 0, 0.0),
    "disk_screened": (lambda: _disk(0.5), 0, 1.9),
    "disk_pure_neumann": (lambda: _disk(1.0), 0, 1.9),
    "box_sphere": (lambda: scenes.box_sphere_scene(), 0, 0.0),
    "cube_faces_leaf16": (lambda: scenes.cube_scene(8, neumann_faces=(0, 3)), 16, 0.0),
    "cube_screened": (lambda: scenes.cube_scene(5, fn="exp_plane", params=(1.0, 0.8, -0.5, 0.6), neumann_faces=(0, 3)),
                      0, 1.25),
    "plate": (lambda: scenes.plate_cube_scene(), 0, 0.0),
    "cube_torus": (lambda: scenes.config3(grid=8, nu=120, nv=48, cube_m=8), 0, 0.0),
}


def _points(sc, n, rng):
    V = sc["vertices"].astype(np.float64)
    lo, hi = V.min(0), V.max(0)
    if sc["dim"] == 3:
        p = lo + (hi - lo) * rng.uniform(0.03, 0.97, (8 * n, 3))
        rho = np.hypot(np.hypot(p[:, 0], p[:, 1]) - 0.5, p[:, 2])
        return p[(rho > 0.24) & (np.linalg.norm(p, axis=1) > 0.45)][:n].astype(np.float32)
    c = 0.5 * (lo + hi)
    if len(V) > 2000 or "koch" in sc.get("name", ""):  # the Koch scenes' domain: between hole and inner disk
        r, t = rng.uniform(0.36, 0.5, n), rng.uniform(0, 2 * np.pi, n)
        return np.c_[r * np.cos(t), r * np.sin(t)].astype(np.float32)
    if "keyhole" in sc.get("name", ""):
        return np.c_[rng.uniform(-1.9, -0.1, n), rng.uniform(-0.9, 0.9, n)].astype(np.float32)
    return (c + 0.25 * (hi - lo) * rng.uniform(-1, 1, (n, 2))).astype(np.float32)


def _both(wost, sc, leaf, sigma, pts, walks, kernel, cap=2048, **kw):
    S = wost.Scene(sc, leaf_size=leaf)
    depth = S.info()["stack_depth"]
    dev = torch.from_numpy(pts).cuda()
    got = [wost.solve(S, dev, walks, 1e-3, 1e-3, cap, seed=3, kernel=kernel, sigma=sigma, stack_depth=d, **kw)
           for d in (0, depth)]
    S.close()
    a, b = got
    assert a["done"] == b["done"] == 1 and a["guard_flags"] == b["guard_flags"] == 0
    assert np.array_equal(a["walks"], b["walks"])
    assert (a["total_steps"], a["capped_walks"], a["steps_run"]) == (b["total_steps"], b["capped_walks"],
                                                                     b["steps_run"])
    np.testing.assert_allclose(a["mean"], b["mean"], rtol=1e-9, atol=1e-12)
    return a


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("n,walks,kernel", [(1, 1, "plain"), (61, 33, "persistent"), (257, 96, "persistent"),
                                            (257, 96, "resumable")])
def test_warp_walks_are_the_one_lane_walks(wost, name, n, walks, kernel):
    make, leaf, sigma = CASES[name]
    sc = make()
    _both(wost, sc, leaf, sigma, _points(sc, n, np.random.default_rng(7)), walks, kernel)


@pytest.mark.parametrize("name", ["koch3", "box_sphere", "cube_faces_leaf16", "cube_torus"])
@pytest.mark.parametrize("n,walks", [(1, 1), (61, 33), (257, 96)])
def test_counting_kernel_runs_the_same_walks_and_counts_all_of_them(wost, name, n, walks):
    """Its searches are the lane's own to their end, whatever the limits."""
    make, leaf, sigma = CASES[name]
    sc = make()
    pts = _points(sc, n, np.random.default_rng(7))
    own = _both(wost, sc, leaf, sigma, pts, walks, "counting")
    ref = _both(wost, sc, leaf, sigma, pts, walks, "persistent")
    assert own["total_steps"] == ref["total_steps"]
    np.testing.assert_allclose(own["mean"], ref["mean"], rtol=1e-9, atol=1e-12)
    S = wost.Scene(sc, leaf_size=leaf)
    given = wost.solve(S, torch.from_numpy(pts).cuda(), walks, 1e-3, 1e-3, 2048, seed=3, kernel="counting",
                       sigma=sigma, stack_depth=S.info()["stack_depth"])
    S.close()
    assert own["counts"] == given["counts"]


def test_warp_walks_from_boundary_points(wost):
    for sc in (scenes.config1(), scenes.box_sphere_scene(data="analytic")):
        sel = np.flatnonzero(sc["flags"] == 1)
        sel = sel[:: max(1, len(sel) // 48)]
        V, P = sc["vertices"], sc["prims"][sel]
        w = np.array([0.3, 0.7]) if sc["dim"] == 2 else np.array([0.2, 0.3, 0.5])
        pts = np.einsum("k,nkd->nd", w, V[P].astype(np.float64)).astype(np.float32)
        nrm = torch.from_numpy(scenes.prim_normals(sc)[sel].astype(np.float32)).cuda()
        on = torch.ones(len(sel), dtype=torch.uint8, device="cuda")
        _both(wost, sc, 0, 0.0, pts, 40, "persistent", normals=nrm, on_neumann=on)


@pytest.mark.parametrize("n,walks", [(300, 64), (900, 400), (3000, 160)])
def test_handed_over_walks_are_the_one_lane_walks(wost, n, walks):
    """Solves larger than one warp per walk: their last walks pass through one
    or more hand-overs (a few thousand walks to more than the GPU's lanes)."""
    for name in ("flower", "koch3", "disk_screened", "box_sphere"):
        make, leaf, sigma = CASES[name]
        sc = make()
        for kernel in ("persistent", "resumable"):
            _both(wost, sc, leaf, sigma, _points(sc, n, np.random.default_rng(11)), walks, kernel, cap=600)


def test_static_solve_and_batch_hand_over_to_warps(wost):
    specs = [CASES[k][0]() for k in ("flower", "koch3", "box_sphere", "cube_torus")]
    S = [wost.Scene(sc) for sc in specs]
    n, walks = [700, 300, 900, 200], [64, 96, 48, 80]
    pts = [torch.from_numpy(_points(sc, k, np.random.default_rng(5))).cuda() for sc, k in zip(specs, n)]
    ref = [wost.solve(s, p, w, 1e-3, 1e-3, 1024, seed=9 + i, kernel="persistent",
                      stack_depth=s.info()["stack_depth"]) for i, (s, p, w) in enumerate(zip(S, pts, walks))]
    hs = wost.wost_solve_batch([s.handle for s in S],
                               [dict(points=p, walks_per_point=w, epsilon=1e-3, r_min=1e-3, max_steps=1024, seed=9 + i)
                                for i, (p, w) in enumerate(zip(pts, walks))])
    for h, r, k in zip(hs, ref, n):
        wost.wost_wait(h, 120)
        mean, _, wd, pr = wost.wost_poll(h, k)
        wost.wost_solve_destroy(h)
        assert np.array_equal(wd, r["walks"]) and pr["total_steps"] == r["total_steps"]
        np.testing.assert_allclose(mean, r["mean"], rtol=1e-9, atol=1e-12)
    for i, (s, p, w, r) in enumerate(zip(S, pts, walks, ref)):
        mean = torch.empty(len(p), device="cuda")
        for _ in range(2):  # the scratch array keeps the first call's contents
            wost.wost_solve_static(s.handle, p, w, 1e-3, 1e-3, 1024, 9 + i, 0, mean)
        np.testing.assert_array_equal(mean.cpu().numpy(), r["mean"].astype(np.float32))
        s.close()


@pytest.mark.parametrize("name", sorted(CASES))
def test_small_query_arrays_get_the_answers_of_large_ones(wost, name):
    """Arrays of few queries (at most 16,384, by query) run one query per warp,
    larger ones one per lane (Q.2 in 3D: always one per warp, checked against
    the oracle elsewhere): the same distances, points, records, hits and samples, bit for
    bit, also for points on vertices and midway between primitives (ties),
    far outside, and not finite."""
    make, leaf, _ = CASES[name]
    sc = make()
    dim = sc["dim"]
    rng = np.random.default_rng(13)
    V = sc["vertices"].astype(np.float64)
    lo, hi = V.min(0), V.max(0)
    k = rng.integers(len(V), size=900)
    P = sc["prims"][rng.integers(len(sc["prims"]), size=900)]
    pts = np.concatenate([lo + (hi - lo) * rng.random((14000, dim)), V[k], V[P].mean(1), 0.5 * (V[P[:, 0]] + V[P[:, 1]]),
                          np.round(lo + (hi - lo) * rng.random((300, dim)), 1), V[k[:100]] * 30.0,
                          np.full((1, dim), np.nan), np.zeros((1, dim))])
    n = len(pts)
    d = rng.normal(size=(n, dim))
    d[::7] = np.eye(dim)[rng.integers(dim, size=len(d[::7]))]  # along an axis
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    x, v, t, r = dev(pts), dev(d), dev(rng.uniform(0.05, 2.0, n)), dev(rng.uniform(0.02, 1.5, n))
    skip = torch.from_numpy(rng.integers(-1, len(sc["prims"]), n).astype(np.int32)).cuda()
    S = wost.Scene(sc, leaf_size=leaf)

    def ask(s):
        m = s.stop - s.start
        return [*wost.wost_query_closest_dirichlet(S.handle, x[s]), wost.wost_query_silhouette(S.handle, x[s], r[s]),
                *wost.wost_query_intersect_neumann(S.handle, x[s], v[s], t[s]),
                *wost.wost_query_intersect_neumann(S.handle, x[s], v[s], t[s], skip=skip[s]),
                *[o[: min(m, 1111)] for o in wost.wost_query_neumann_sample(S.handle, x[s], r[s], 5, 1, 2)]]

    assert n > 16384
    whole = ask(slice(0, n))
    parts = [ask(slice(a, min(a + 1111, n))) for a in range(0, n, 1111)]
    for i, w in enumerate(whole):
        # (a sample's random numbers are keyed by its index in the array: the first part only)
        got = parts[0][i] if i >= len(whole) - 3 else torch.cat([p[i] for p in parts])
        np.testing.assert_array_equal(got.cpu().numpy(), w.cpu().numpy(), err_msg=f"{name}: output {i}")
    S.close()

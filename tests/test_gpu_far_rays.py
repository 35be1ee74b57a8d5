"""Q.3 for origins far outside the scene: a small array of rays (one ray per
warp) gets the hits of a large one (one per lane), bit for bit.  The rounding
of a box test grows with the distance of the origin, and rays aimed at edges,
vertices and faces of the boundary show it."""
import numpy as np
import pytest

from paper_2302_11815_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCENES = {
    "flower": lambda: scenes.config1(n_points=1),
    "koch4": lambda: scenes.config2(grid=8, level=4),
    "box_sphere": lambda: scenes.box_sphere_scene(),
    "cube": lambda: scenes.cube_scene(8, neumann_faces=(0, 3)),
    "cube_torus": lambda: scenes.config3(grid=4, nu=120, nv=48),
}


@pytest.fixture(scope="module")
def wost():
    from paper_2302_11815_gb300 import build as libbuild
    from paper_2302_11815_gb300 import wost as w

    assert torch.cuda.is_available()
    libbuild.build()
    w.load()
    return w


@pytest.mark.parametrize("name", sorted(SCENES))
@pytest.mark.parametrize("far", [30, 300, 1000, 10000, 100000])
def test_rays_from_far_away_hit_the_same_records(wost, name, far):
    sc = SCENES[name]()
    dim = sc["dim"]
    rng = np.random.default_rng(2)
    V = sc["vertices"].astype(np.float64)
    P = V[sc["prims"][sc["flags"] == 1][:, :dim]]
    size = np.abs(V).max()
    n, part = 20000, 1000
    pick = P[rng.integers(len(P), size=n)]
    w = rng.dirichlet(np.ones(dim), n)
    w[: n // 4] = np.eye(dim)[0]  # a vertex
    w[n // 4: n // 2] = [0.5, 0.5] + [0.0] * (dim - 2)  # an edge (2D: the middle)
    d = rng.normal(size=(n, dim))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    o, v = dev(np.einsum("nk,nkd->nd", w, pick) - d * size * far), dev(d)
    reach = dev(size * far * rng.uniform(1.0, 1.5, n) + 2)
    S = wost.Scene(sc)
    whole = wost.wost_query_intersect_neumann(S.handle, o, v, reach)
    parts = [wost.wost_query_intersect_neumann(S.handle, o[a: a + part], v[a: a + part], reach[a: a + part])
             for a in range(0, n, part)]
    S.close()
    assert int(whole[0].sum()) > n // 2
    for i, what in enumerate(("hit", "t", "prim")):
        np.testing.assert_array_equal(torch.cat([p[i] for p in parts]).cpu().numpy(), whole[i].cpu().numpy(),
                                      err_msg=f"{name} {far}: {what}")

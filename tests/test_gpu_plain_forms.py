"""The plain kernel's two forms in 3D, silhouette searches joint or each its
lane's own (by the number of candidates), run the walks of the persistent
kernel with given limits."""
import numpy as np
import pytest

from paper_2302_11815_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# silhouette candidates: 108, 1,584 (below the line of 8,192), 17,280
SCENES = {
    "cube": (lambda: scenes.cube_scene(4, neumann_faces=(0, 3)), 0.0),
    "cube_fine_screened": (lambda: scenes.cube_scene(16, fn="exp_plane", params=(1.0, 0.8, -0.5, 0.6),
                                                     neumann_faces=(0, 3)), 1.25),
    "cube_torus": (lambda: scenes.config3(grid=8, nu=120, nv=48, cube_m=8), 0.0),
    "cube_torus_screened": (lambda: scenes.config3(grid=8, nu=120, nv=48, cube_m=8), 0.6),
}


@pytest.mark.parametrize("name", sorted(SCENES))
def test_plain_kernel_runs_the_same_walks(name):
    from paper_2302_11815_gb300 import build as libbuild
    from paper_2302_11815_gb300 import wost

    assert torch.cuda.is_available()
    libbuild.build()
    wost.load()
    make, sigma = SCENES[name]
    p = np.random.default_rng(7).uniform(-0.95, 0.95, (4000, 3))
    rho = np.hypot(np.hypot(p[:, 0], p[:, 1]) - 0.5, p[:, 2])
    pts = p[rho > 0.24][:257].astype(np.float32)
    S = wost.Scene(make())
    assert len(pts) * 96 > 16384  # (fewer walks would run one per warp)
    got = wost.solve(S, pts, 96, 1e-3, 1e-3, 2048, seed=3, kernel="plain", sigma=sigma)
    lim = wost.solve(S, pts, 96, 1e-3, 1e-3, 2048, seed=3, kernel="plain", sigma=sigma,
                     stack_depth=S.info()["stack_depth"])
    ref = wost.solve(S, pts, 96, 1e-3, 1e-3, 2048, seed=3, kernel="persistent", sigma=sigma,
                     stack_depth=S.info()["stack_depth"])
    S.close()
    for r in (got, lim):
        assert np.array_equal(r["walks"], ref["walks"]) and r["total_steps"] == ref["total_steps"]
        assert r["guard_flags"] == 0 and r["capped_walks"] == ref["capped_walks"]
        np.testing.assert_allclose(r["mean"], ref["mean"], rtol=1e-9, atol=1e-12)

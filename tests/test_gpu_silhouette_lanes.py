"""Q.2 in 3D by one warp per query and by one lane per query: the same
distances, bit for bit, also at points on vertices and midway between
primitives (ties, grazing directions), far outside, and not finite.  (The
call's own choice between the two is by size: both launchers are called here.)"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2302_11815_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

SCENES = {
    "box_sphere": (lambda: scenes.box_sphere_scene(), 0),
    "box_sphere_leaf1": (lambda: scenes.box_sphere_scene(m=6, n_lat=16, n_lon=32), 1),
    "cube": (lambda: scenes.cube_scene(4, neumann_faces=(0, 3)), 0),
    "cube_faces_leaf16": (lambda: scenes.cube_scene(8, neumann_faces=(0, 3)), 16),
    "cube_fine": (lambda: scenes.cube_scene(16, neumann_faces=(0, 3)), 0),
    "plate": (lambda: scenes.plate_cube_scene(), 0),
    "box_sphere_coarse": (lambda: scenes.box_sphere_scene(m=2, n_lat=8, n_lon=16), 0),
    "cube_torus": (lambda: scenes.config3(grid=4, nu=120, nv=48, cube_m=8), 0),
}


@pytest.fixture(scope="module")
def wost():
    from paper_2302_11815_gb300 import build as libbuild
    from paper_2302_11815_gb300 import wost as w

    assert torch.cuda.is_available()
    libbuild.build()
    w.load()
    return w


@pytest.fixture(scope="module")
def ask(wost, tmp_path_factory):
    from paper_2302_11815_gb300 import build as libbuild

    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    so = str(tmp_path_factory.mktemp("lane_query") / "liblanequery.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-w", "-I" + inc, "-I" + libbuild.CSRC,
                    "-I" + os.path.join(libbuild.ROOT, "include"), os.path.join(HERE, "lane_query.cpp"), "-o", so,
                    libbuild.LIB, "-Wl,-rpath," + os.path.dirname(libbuild.LIB)], check=True)
    fn = C.CDLL(so).lane_query_silhouette
    fn.argtypes = [C.c_void_p, C.c_int64, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]

    def ask(scene, x, r, per_warp):
        out = torch.empty(len(x), device="cuda")
        torch.cuda.synchronize()
        assert fn(scene, len(x), x.data_ptr(), r.data_ptr(), out.data_ptr(), per_warp) == 0
        torch.cuda.synchronize()
        return out.cpu().numpy()

    return ask


def _queries(sc, n, rng):
    V = sc["vertices"].astype(np.float64)
    lo, hi = V.min(0), V.max(0)
    k = rng.integers(len(V), size=1500)
    P = sc["prims"][rng.integers(len(sc["prims"]), size=1500)]
    x = np.concatenate([lo + (hi - lo) * rng.random((n, 3)), V[k], V[P].mean(1), 0.5 * (V[P[:, 0]] + V[P[:, 1]]),
                        np.round(lo + (hi - lo) * rng.random((500, 3)), 1), V[k[:300]] * 30.0, V[k[:300]] * 1000.0,
                        np.full((1, 3), np.nan), np.zeros((1, 3))]).astype(np.float32)
    r = rng.uniform(0.02, 1.5, len(x))
    r[::5] = rng.uniform(1.5, 4000.0, len(r[::5]))
    r[::97] = np.inf
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    return dev(x), dev(r)


@pytest.mark.parametrize("name", sorted(SCENES))
def test_one_warp_and_one_lane_per_query_agree(wost, ask, name):
    make, leaf = SCENES[name]
    sc = make()
    S = wost.Scene(sc, leaf_size=leaf)
    x, r = _queries(sc, 20000, np.random.default_rng(13))
    np.testing.assert_array_equal(ask(S.handle, x, r, 1), ask(S.handle, x, r, 0), err_msg=name)
    S.close()


@pytest.mark.parametrize("name,n", [("cube", 131072), ("cube", 131073), ("plate", 131073), ("box_sphere_coarse", 131073),
                                    ("box_sphere_coarse", 1048577), ("cube_fine", 1048577)])
def test_arrays_on_both_sides_of_the_size_rule(wost, ask, name, n):
    """Up to 256 candidates and more than 131,072 queries, or up to 384 and
    more than 1,048,576: one lane each."""
    sc = SCENES[name][0]()
    S = wost.Scene(sc)
    x, r = _queries(sc, n, np.random.default_rng(3))
    x, r = x[-n:].contiguous(), r[-n:].contiguous()
    got = wost.wost_query_silhouette(S.handle, x, r).cpu().numpy()
    np.testing.assert_array_equal(got, ask(S.handle, x, r, 1))
    np.testing.assert_array_equal(got, ask(S.handle, x, r, 0))
    S.close()

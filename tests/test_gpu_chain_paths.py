"""Ways into and out of a chain of launches: saved walks taken up by the chain,
more than one hand-over in the static solve, cancelling, sets of resources that
solves of several sizes, threads and streams use in turn, and launches that
find no memory to hand walks over in.  Walks are those of the one-lane kernels
(a solve that gives its traversal limits), as in test_gpu_warp_walks.py."""
import ctypes as C
import os
import shutil
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

from paper_2302_11815_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

SCENES = {
    "flower": lambda: scenes.config1(n_points=1),
    "koch3": lambda: scenes.config2(grid=8, level=3),
    "box_sphere": lambda: scenes.box_sphere_scene(),
}


@pytest.fixture(scope="module")
def wost():
    from paper_2302_11815_gb300 import build as libbuild
    from paper_2302_11815_gb300 import wost as w

    assert torch.cuda.is_available()
    libbuild.build()
    w.load()
    return w


def _points(name, n, seed=11):
    rng = np.random.default_rng(seed)
    if name == "box_sphere":
        p = rng.uniform(-0.95, 0.95, (8 * n, 3))
        return p[np.linalg.norm(p, axis=1) > 0.45][:n].astype(np.float32)
    r, t = rng.uniform(0.36, 0.5, n), rng.uniform(0, 2 * np.pi, n)
    return np.c_[r * np.cos(t), r * np.sin(t)].astype(np.float32)


def _one_lane(wost, S, pts, walks, cap, seed, **kw):
    return wost.solve(S, pts, walks, 1e-3, 1e-3, cap, seed=seed, kernel="persistent",
                      stack_depth=S.info()["stack_depth"], **kw)


def _same(got, ref):
    assert np.array_equal(got["walks"], ref["walks"])
    assert got["total_steps"] == ref["total_steps"] and got["guard_flags"] == 0
    np.testing.assert_allclose(got["mean"], ref["mean"], rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("name", sorted(SCENES))
@pytest.mark.parametrize("n,walks,iters", [(61, 33, 3), (300, 160, 1), (1500, 100, 5), (1500, 100, 1000)])
def test_a_wait_takes_up_the_walks_that_an_advanced_solve_saved(wost, name, n, walks, iters):
    S = wost.Scene(SCENES[name]())
    pts = _points(name, n)
    ref = _one_lane(wost, S, pts, walks, 900, 5)
    h = wost.wost_solve(S.handle, pts, walks, 1e-3, 1e-3, 900, seed=5, kernel="resumable")
    wost.wost_solve_advance(h, iters)
    wost.wost_wait(h, 60)
    mean, _, wd, pr = wost.wost_poll(h, n)
    wost.wost_solve_destroy(h)
    _same(dict(pr, mean=mean, walks=wd), ref)
    assert pr["steps_run"] == pr["total_steps"]
    S.close()


@pytest.mark.parametrize("name,n,walks", [("flower", 3000, 64), ("koch3", 800, 100), ("box_sphere", 40000, 8)])
def test_static_solves_with_several_hand_overs(wost, name, n, walks):
    """More walks than twice the fixed array's slots: two hand-overs."""
    S = wost.Scene(SCENES[name]())
    pts = torch.from_numpy(_points(name, n)).cuda()
    ref = _one_lane(wost, S, pts, walks, 900, 6)
    mean = torch.empty(n, device="cuda")
    wost.wost_solve_static(S.handle, pts, walks, 1e-3, 1e-3, 900, 6, 0, mean)
    np.testing.assert_array_equal(mean.cpu().numpy(), ref["mean"].astype(np.float32))
    S.close()


def test_static_solves_in_a_graph(wost):
    """Captured after a first call of another size, replayed on other points."""
    S = wost.Scene(SCENES["flower"]())
    a, b = (torch.from_numpy(_points("flower", 3000, s)).cuda() for s in (1, 2))
    pts, mean = a.clone(), torch.empty(3000, device="cuda")
    wost.wost_solve_static(S.handle, pts[:10].contiguous(), 4, 1e-3, 1e-3, 900, 6, 0, mean)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        wost.wost_solve_static(S.handle, pts, 64, 1e-3, 1e-3, 900, 6, 0, mean, stream=torch.cuda.current_stream())
    for x in (a, b, a):
        pts.copy_(x)
        graph.replay()
        torch.cuda.synchronize()
        ref = _one_lane(wost, S, x, 64, 900, 6)
        np.testing.assert_array_equal(mean.cpu().numpy(), ref["mean"].astype(np.float32))
    S.close()


@pytest.mark.parametrize("kernel", ["persistent", "resumable"])
def test_cancelling_while_a_chain_runs(wost, kernel):
    S = wost.Scene(scenes.config2(grid=8, level=4))
    pts = _points("koch4", 900)
    ref = _one_lane(wost, S, pts[:64], 16, 512, 9)
    n, walks = len(pts), 4096
    h = wost.wost_solve(S.handle, pts, walks, 1e-4, 1e-4, 4096, seed=8, kernel=kernel)
    waiter = threading.Thread(target=wost.wost_wait_status, args=(h, -1.0))
    waiter.start()  # (a resumable solve advances while it is waited for)
    time.sleep(0.02)
    wost.wost_cancel(h)
    waiter.join(120)
    assert not waiter.is_alive()
    assert wost.wost_wait_status(h, 10.0) == wost.ERR_CANCELLED
    mean, _, wd, pr = wost.wost_poll(h, n)
    wost.wost_solve_destroy(h)
    assert pr["done"] == 1 and 0 < int(wd.sum()) < n * walks and np.isfinite(mean).all()
    # the set of resources goes on to the next solve
    got = wost.solve(S, pts[:64], 16, 1e-3, 1e-3, 512, seed=9, kernel=kernel)
    _same(got, ref)
    S.close()


def test_solves_of_several_sizes_threads_and_streams_on_one_scene(wost):
    S = wost.Scene(SCENES["flower"]())
    sizes = [(40, 8), (3000, 64), (7, 300), (900, 200), (1, 1), (2000, 30)]
    ref = {s: _one_lane(wost, S, _points("flower", s[0], s[1]), s[1], 900, 3) for s in sizes}
    failed = []

    def work(i):
        try:
            stream = torch.cuda.Stream() if i % 2 else None
            for j in range(12):
                s = sizes[(i + j * (1 + i)) % len(sizes)]
                pts = _points("flower", s[0], s[1])
                kernel = ("persistent", "resumable", "plain")[(i + j) % 3]
                if j % 4 == 3:
                    pts = torch.from_numpy(pts).cuda()
                    torch.cuda.synchronize()
                _same(wost.solve(S, pts, s[1], 1e-3, 1e-3, 900, seed=3, kernel=kernel, stream=stream), ref[s])
        except Exception as e:  # noqa: BLE001
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(300)
    assert not failed and not any(t.is_alive() for t in threads), failed[:2]
    S.close()


@pytest.mark.parametrize("sigma", [0.0, 0.7])
@pytest.mark.parametrize("n,walks", [(1, 3), (40, 60), (900, 64), (2500, 150)])
def test_batches_hand_their_last_walks_over(wost, sigma, n, walks):
    """Both forms of the batched kernel (screened, Poisson only), from fewer
    walks than a launch hands over at once to more than its lanes."""
    names = ["flower", "box_sphere", "koch3"]
    S = [wost.Scene(SCENES[k]()) for k in names]
    pts = [_points(k, n + 7 * i) for i, k in enumerate(names)]
    ref = [_one_lane(wost, s, p, walks, 900, 4 + i, sigma=sigma) for i, (s, p) in enumerate(zip(S, pts))]
    hs = wost.wost_solve_batch([s.handle for s in S], [dict(points=p, walks_per_point=walks, epsilon=1e-3, r_min=1e-3,
                                                            max_steps=900, seed=4 + i, sigma=sigma)
                                                       for i, p in enumerate(pts)])
    for h, p, r in zip(hs, pts, ref):
        wost.wost_wait(h, 120)
        mean, _, wd, pr = wost.wost_poll(h, len(p))
        _same(dict(pr, mean=mean, walks=wd), r)
    for h in hs:
        wost.wost_solve_destroy(h)
    for s in S:
        s.close()


_WITHOUT_SLOTS = """
import ctypes as C, sys
import numpy as np, torch
from paper_2302_11815_gb300 import scenes, wost
lib = wost.load(sys.argv[1])
lib.fault_between.argtypes = [C.c_size_t, C.c_size_t]
sys.path.insert(0, "tests")
from test_gpu_chain_paths import SCENES, _one_lane, _points, _same
names = ["flower", "koch3", "box_sphere"]
S = [wost.Scene(SCENES[k]()) for k in names]
pts = [_points(k, 900) for k in names]
sig = [0.0, 0.0, 0.7]
ref = [_one_lane(wost, s, p, 64, 900, 4, sigma=q) for s, p, q in zip(S, pts, sig)]
lib.fault_between(1 << 20, 7 << 20)  # the slots (a resumable solve's own take 8 MB)
for kernel in ("persistent", "resumable"):
    for s, p, r, q in zip(S, pts, ref, sig):
        was = lib.fault_count()
        got = wost.solve(s, p, 64, 1e-3, 1e-3, 900, seed=4, kernel=kernel, sigma=q)
        assert kernel == "resumable" or lib.fault_count() > was
        _same(got, r)
for mixed in (sig, [0.0] * 3):  # the screened form of the batched kernel, and the other
    was = lib.fault_count()
    hs = wost.wost_solve_batch([s.handle for s in S], [dict(points=p, walks_per_point=64, epsilon=1e-3, r_min=1e-3,
                                                            max_steps=900, seed=4, sigma=q)
                                                       for p, q in zip(pts, mixed)])
    assert lib.fault_count() > was
    for h, s, p, r, q in zip(hs, S, pts, ref, mixed):
        wost.wost_wait(h, 60)
        mean, _, wd, pr = wost.wost_poll(h, len(p))
        wost.wost_solve_destroy(h)
        _same(dict(pr, mean=mean, walks=wd), r if q == sig[S.index(s)] else _one_lane(wost, s, p, 64, 900, 4, sigma=q))
print("WITHOUT SLOTS OK")
"""


def test_without_memory_for_slots_the_walks_are_the_same(wost, tmp_path):
    """The host code with a cudaMalloc that refuses the slots' sizes, in a
    process of its own."""
    from paper_2302_11815_gb300 import build as libbuild

    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    inc = ["-I" + os.path.join(cuda, "include"), "-I" + libbuild.CSRC, "-I" + os.path.join(libbuild.ROOT, "include")]
    capi, fault, so = (str(tmp_path / f) for f in ("capi.o", "fault.o", "libwost_fault.so"))
    gxx = ["g++", "-O1", "-std=c++17", "-fPIC", "-w", *inc, "-c"]
    subprocess.run([*gxx, "-DcudaMalloc=faulty_cudaMalloc", os.path.join(libbuild.CSRC, "wost_capi.cpp"), "-o", capi],
                   check=True)
    subprocess.run([*gxx, os.path.join(HERE, "alloc_fault.cpp"), "-o", fault], check=True)
    objs = [os.path.join(libbuild.BUILD, os.path.basename(s) + ".o") for s in libbuild._sources()]
    assert all(os.path.exists(o) for o in objs)
    objs = [o for o in objs if "wost_capi" not in o]
    subprocess.run([nvcc, *libbuild.ARCH, "-shared", "-o", so, capi, fault, *objs], check=True)
    r = subprocess.run([sys.executable, "-c", _WITHOUT_SLOTS, so], cwd=libbuild.ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "WITHOUT SLOTS OK" in r.stdout, r.stdout + r.stderr

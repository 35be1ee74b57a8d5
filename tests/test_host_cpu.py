"""The host side of the C ABI without a device: wost_capi.cpp linked against
hostsim.cpp, which stands in for the CUDA runtime and the kernel launchers
and records how streams, memory and launches are used."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2302_11815_gb300 import build as libbuild
from paper_2302_11815_gb300 import scenes, wost

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def simlib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    out = tmp_path_factory.mktemp("hostsim")
    objs = []
    src = [os.path.join(libbuild.CSRC, f) for f in ("wost_capi.cpp", "scene_build.cpp", "scene_check.cpp")]
    for s in [*src, os.path.join(HERE, "hostsim.cpp")]:
        objs.append((s, str(out / (os.path.basename(s) + ".o"))))
    procs = [subprocess.Popen(["g++", "-O1", "-std=c++17", "-fPIC", "-w", "-I" + inc, "-I" + libbuild.CSRC, "-I" +
                               os.path.join(libbuild.ROOT, "include"), "-c", s, "-o", o]) for s, o in objs]
    assert all(p.wait() == 0 for p in procs)
    path = str(out / "libhostsim.so")
    # (its own cuda* functions, whatever else the process has loaded)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", path, *[o for _, o in objs], "-lpthread"], check=True)
    lib = C.CDLL(path)
    for name, argt in wost._SIGS.items():
        if hasattr(lib, name):
            getattr(lib, name).argtypes = argt
            getattr(lib, name).restype = C.c_int
    lib.wost_last_error.restype = C.c_char_p
    lib.sim_log.restype = C.c_char_p
    lib.sim_used.restype = C.c_size_t
    lib.sim_reset.argtypes = lib.sim_limit.argtypes = [C.c_size_t]
    return lib


@pytest.fixture
def sim(simlib, monkeypatch):
    """The stand-in in place of the library."""
    monkeypatch.setattr(wost, "_lib", simlib)
    simlib.sim_reset(1 << 40)
    return simlib


def _log(sim):
    return sim.sim_log().decode().split("\n")[:-1]


def _stream(sim):
    s = C.c_void_p()
    assert sim.cudaStreamCreateWithFlags(C.byref(s), 0) == 0
    return s.value


def _solve(scene, n=64, walks=4, kernel="persistent", **kw):
    return wost.wost_solve(scene.handle, np.zeros((n, scene.dim), np.float32), walks, 1e-3, 1e-3, 256, 1, 0, kernel,
                           **kw)


def test_destroy_leaves_a_stream_alone_that_the_caller_has_destroyed(sim):
    """A handle whose work has completed touches its stream no more: a
    resumable solve that was never advanced, and a finished one."""
    S = wost.Scene(scenes.config1(n_points=1))
    for kernel in ("resumable", "persistent", "plain"):
        s = _stream(sim)
        h = _solve(S, kernel=kernel, stream=s)
        if kernel != "resumable":
            wost.wost_wait(h)
        sim.cudaStreamDestroy(C.c_void_p(s))
        wost.wost_solve_destroy(h)
        assert sim.sim_bad() == 0, kernel
    S.close()


@pytest.mark.parametrize("kernel", ["persistent", "resumable"])
def test_destroy_waits_for_reads_of_accumulators_handed_out(sim, kernel):
    """A solve's memory goes to the next solve of its scene at once: reads that
    the caller enqueued through the pointers it was given must be over."""
    S = wost.Scene(scenes.config1(n_points=1))
    h = _solve(S, kernel=kernel)
    wost.wost_wait(h)
    wost.wost_solve_destroy(h)
    assert "device synchronised" not in _log(sim)
    h = _solve(S, kernel=kernel)
    wost.wost_wait(h)
    assert all(wost.wost_solve_device_accumulators(h))
    wost.wost_solve_destroy(h)
    assert _log(sim)[-1] == "device synchronised"
    S.close()


def _finished(S, n, walks=4, kernel="persistent"):
    h = _solve(S, n, walks, kernel)
    wost.wost_wait(h)
    wost.wost_solve_destroy(h)


def _batch(S, n, walks):
    hs = wost.wost_solve_batch([S.handle], [dict(points=np.zeros((n, S.dim), np.float32), walks_per_point=walks,
                                                 epsilon=1e-3, r_min=1e-3, max_steps=256, seed=1)])
    for h in hs:
        wost.wost_wait(h)
        wost.wost_solve_destroy(h)


@pytest.mark.parametrize("what", ["scene", "solve", "counting", "resumable", "batch"])
def test_memory_that_is_short_comes_from_other_scenes_idle_sets(sim, what):
    """A finished solve's memory stays with its scene for the next solve, until
    an allocation of the library finds none: whichever scene's it is."""
    spec = scenes.config1(n_points=1)
    A, B = wost.Scene(spec), wost.Scene(spec)
    _finished(A, 200000)
    sim.sim_limit(sim.sim_used())  # nothing is left but A's idle set
    if what == "scene":
        wost.Scene(spec).close()
    elif what == "batch":
        _batch(B, 1000, 4)
    else:
        _finished(B, 1000, kernel="persistent" if what == "solve" else what)
    A.close()
    B.close()


def test_idle_memory_of_all_scenes_is_bounded(sim):
    spec = scenes.config1(n_points=1)
    before = sim.sim_used()
    S = [wost.Scene(spec) for _ in range(12)]
    held = sim.sim_used()
    for s in S:
        _finished(s, 600000, 1)  # some 40 MB each, 480 in all
    assert sim.sim_used() - held <= 256 << 20
    # the last scenes' sets are those that are left
    used = sim.sim_used()
    _finished(S[-1], 600000, 1)
    assert sim.sim_used() == used
    for s in S:
        s.close()
    assert sim.sim_used() == before


@pytest.mark.parametrize("kernel,want", [("persistent", ["persistent"]), ("resumable", ["resume 2048"] * 4),
                                         ("batch", ["batch 2d without slots"])])
def test_without_memory_for_hand_overs_the_walks_stay(sim, kernel, want):
    S = wost.Scene(scenes.config1(n_points=1))
    sim.sim_limit(sim.sim_used() + (1 << 20))  # (the stand-in's slots take 6 MB)
    if kernel == "batch":
        _batch(S, 64, 400)
    else:
        _finished(S, 64, 400, kernel)
    assert _log(sim) == want
    S.close()


def test_a_batch_keeps_its_slots_for_the_next_one(sim):
    """The slots come from the resources that the scenes keep: a second batch
    of the same size takes no more memory than the first left, its job tables
    and counters aside."""
    S = [wost.Scene(scenes.config1(n_points=1)), wost.Scene(scenes.cube_scene(2, neumann_faces=(0,)))]

    def batch():
        hs = wost.wost_solve_batch([s.handle for s in S],
                                   [dict(points=np.zeros((64, s.dim), np.float32), walks_per_point=400, epsilon=1e-3,
                                         r_min=1e-3, max_steps=256, seed=1) for s in S])
        for h in hs:
            wost.wost_wait(h)
        used = sim.sim_used()
        for h in hs:
            wost.wost_solve_destroy(h)
        return used

    used = batch()
    sim.sim_limit(sim.sim_used() + (1 << 16))  # (a dimension's slots take 6 MB in the stand-in)
    assert batch() == used
    assert _log(sim) == ["batch 2d", "batch 3d"] * 2
    for s in S:
        s.close()


def _tune(sim, S, n, walks, to_go):
    """wost_scene_autotune (the stand-in's device memory is host memory)."""
    pts = np.zeros((n, S.dim), np.float32)
    r = wost.wost_tune_result()
    sim.sim_to_go(to_go)
    assert sim.wost_scene_autotune(S.handle, pts.ctypes.data, n, walks, 1e-3, 1e-3, 256, C.byref(r)) == 0
    assert r.n_tried == 8 and list(r.tried_lanes) == [1] * 4 + [8] * 4
    assert S.info()["lanes_per_walk"] == r.lanes_per_walk
    return r


def test_tuner_times_what_a_solve_runs(sim):
    """A sample whose walks do not last the timed launches is timed as whole
    solves (the stand-in's 8 lanes are twice as fast per launch and half as
    fast for a solve)."""
    S = wost.Scene(scenes.config1(n_points=1))
    r = _tune(sim, S, 64, 400, 1)
    assert r.lanes_per_walk == 1 and _log(sim)[-8:] == ["chain"] * 4 + ["persistent, 8 lanes"] * 4
    assert r.steps_per_second == max(r.tried_steps_per_second) > 0
    sim.sim_reset(1 << 40)
    r = _tune(sim, S, 64, 400, 10**6)
    assert r.lanes_per_walk == 8 and _log(sim) == ["resume 256"] * 24
    S.close()


def test_small_solves_of_a_scene_tuned_to_teams_run_one_walk_per_warp(sim):
    S = wost.Scene(scenes.config1(n_points=1))
    assert _tune(sim, S, 64, 400, 10**6).lanes_per_walk == 8
    for walks, kw, want in [(256, {}, "one per warp"), (257, {}, "persistent, 8 lanes"),
                            (256, dict(lanes_per_walk=8), "persistent, 8 lanes"),
                            (256, dict(stack_depth=9), "persistent, 8 lanes")]:
        wost.wost_solve_destroy(_solve(S, 64, walks, **kw))
        assert _log(sim)[-1] == want, (walks, kw)
    S.close()


def _resumable(S, cap, walks=4):
    return wost.wost_solve(S.handle, np.zeros((64, S.dim), np.float32), walks, 1e-3, 1e-3, cap, 1, 0, "resumable")


@pytest.mark.parametrize("cap,walks,limit,want", [
    # no limit: the chain of launches that runs every walk to its end
    (256, 4, -1.0, ["chain"]),
    (1 << 20, 4, -1.0, ["chain"]),
    # the whole chain ends within the limit whatever the walks do (0.02, 66 s)
    (256, 4, 0.5, ["chain"]),
    (1 << 20, 4, 100.0, ["chain"]),
    # it does not (862 s), but the walks that the stand-in's 2,048 lanes hold
    # end within a quarter of the limit (4.6 s)
    (1 << 16, 4096, 30.0, ["chain"]),
    # ... or does not: bounded launches until all are drawn, then the last
    # five's chain, which ends in 3.3 s
    (1 << 16, 4096, 10.0, ["resume 2048"] * 3 + ["chain from saved walks"]),
    (1 << 16, 4096, 3.0, ["resume 2048"] * 4),
    (1 << 20, 4, 5.0, ["resume 2048"] * 4),
    # a bounded launch would run such walks to their ends as well
    (2048, 4096, 0.1, ["chain"]),
    (2049, 4096, 0.1, ["resume 2048"] * 4),
])
def test_a_limited_wait_starts_no_chain_that_outlasts_it(sim, cap, walks, limit, want):
    S = wost.Scene(scenes.config1(n_points=1))
    h = _resumable(S, cap, walks)
    wost.wost_wait(h, limit)
    assert _log(sim) == want
    wost.wost_solve_destroy(h)
    S.close()


@pytest.mark.parametrize("cap,limit,launched", [(1 << 16, 0.02, "resume 2048"), (256, 0.1, "chain")])
def test_destroying_after_a_timeout_drops_the_walks_not_drawn(sim, cap, limit, launched):
    S = wost.Scene(scenes.config1(n_points=1))
    h = _resumable(S, cap)
    sim.sim_hold(1)  # launches stay in flight
    with pytest.raises(wost.WostError) as e:
        wost.wost_wait(h, limit)
    assert e.value.status == wost.ERR_TIMEOUT
    assert _log(sim) == [launched]
    wost.wost_solve_destroy(h)
    assert _log(sim) == [launched, "waiting, cancelled"]
    sim.sim_hold(0)
    h = _resumable(S, 256)  # the next solve has the set's flag cleared
    wost.wost_wait(h)
    wost.wost_solve_destroy(h)
    S.close()


def test_an_advanced_solve_ends_in_the_chain_over_its_saved_walks(sim):
    S = wost.Scene(scenes.config1(n_points=1))
    for limit in (-1.0, 5.0):
        sim.sim_reset(1 << 40)
        h = _resumable(S, 256)
        for _ in range(3):  # (the stand-in's third launch draws the last walk)
            wost.wost_solve_advance(h, 7)
        wost.wost_wait(h, limit)
        assert _log(sim) == ["resume 7"] * 3 + ["chain from saved walks"]
        wost.wost_solve_destroy(h)
    S.close()


@pytest.mark.parametrize("failing", [1, 2, 3, 4, 5])
def test_a_batch_that_fails_leaves_nothing_in_flight(sim, failing):
    """Its solves' memory goes back at once: both launches, on the call's
    stream and on the 3D one's, have to be over.  (Records of the call: copies,
    start, fork, join, end.)"""
    S = [wost.Scene(scenes.config1(n_points=1)), wost.Scene(scenes.cube_scene(2, neumann_faces=(0,)))]
    req = [dict(points=np.zeros((64, s.dim), np.float32), walks_per_point=400, epsilon=1e-3, r_min=1e-3, max_steps=256,
                seed=1) for s in S]
    sim.sim_fail_record(failing)
    with pytest.raises(wost.WostError):
        wost.wost_solve_batch([s.handle for s in S], req)
    assert _log(sim) == (["batch 2d", "batch 3d"] if failing > 3 else [])
    assert sim.sim_busy() == 0
    for s in S:
        s.close()


def test_destroying_without_host_memory_gives_the_resources_up(sim):
    """Nothing that destroy does may throw: a set that cannot be kept is freed
    (in a child process, which would be aborted)."""
    used = sim.sim_used()
    S = wost.Scene(scenes.config1(n_points=1))
    T = wost.Scene(scenes.config1(n_points=1))
    _finished(S, 64)
    h = _solve(T)
    wost.wost_wait(h)
    pid = os.fork()
    if pid == 0:
        code = 1
        try:
            sim.sim_refuse_new(1)
            ok = sim.wost_solve_destroy(h) == 0 and sim.wost_scene_destroy(S.handle) == 0
            ok = ok and sim.wost_scene_destroy(T.handle) == 0 and sim.sim_used() == used
            code = 0 if ok else 2
        finally:
            os._exit(code)
    assert os.waitpid(pid, 0)[1] == 0
    wost.wost_solve_destroy(h)
    S.close()
    T.close()

"""wost_solve starts its walks and returns, also as the first call of a process,
when none of the kernels of its chain is loaded yet: the solve can be polled
and cancelled while it runs."""
import subprocess
import sys

import pytest

from paper_2302_11815_gb300 import build as libbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_FIRST = """
import sys, time
import numpy as np, torch
from paper_2302_11815_gb300 import scenes, wost
dim, sigma, kernel = int(sys.argv[1]), float(sys.argv[2]), sys.argv[3]
wost.load()
torch.zeros(1, device="cuda")
rng = np.random.default_rng(1)
if dim == 2:
    S = wost.Scene(scenes.config2(grid=8, level=4))
    r, t = rng.uniform(0.36, 0.5, 2000), rng.uniform(0, 2 * np.pi, 2000)
    pts, walks, cap = np.c_[r * np.cos(t), r * np.sin(t)], 400, 16384
else:
    S = wost.Scene(scenes.config3(grid=4, nu=120, nv=48))
    p = rng.uniform(-0.95, 0.95, (200000, 3))
    pts, walks, cap = p[np.hypot(np.hypot(p[:, 0], p[:, 1]) - 0.5, p[:, 2]) > 0.24][:100000], 32, 1024
pts = pts.astype(np.float32)
t0 = time.perf_counter()
h = wost.wost_solve(S.handle, pts, walks, 1e-4, 1e-4, cap, seed=7, kernel=kernel, sigma=sigma)
if kernel == "resumable":
    wost.wost_wait_status(h, 1e-9)
t1 = time.perf_counter()
done = wost.wost_poll(h, len(pts))[3]["done"]
wost.wost_wait(h)
t2 = time.perf_counter()
wost.wost_solve_destroy(h)
print("RETURNED", done, t1 - t0, t2 - t0)
"""


@pytest.mark.parametrize("dim,sigma,kernel", [(2, 0.0, "persistent"), (2, 0.01, "persistent"), (3, 0.0, "persistent"),
                                              (3, 0.01, "persistent"), (2, 0.0, "resumable")])
def test_the_first_solve_of_a_process_returns_while_its_walks_run(dim, sigma, kernel):
    assert torch.cuda.is_available()
    libbuild.build()
    r = subprocess.run([sys.executable, "-c", _FIRST, str(dim), str(sigma), kernel], cwd=libbuild.ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "RETURNED" in r.stdout, r.stdout + r.stderr
    done, call, whole = (float(x) for x in r.stdout.split("RETURNED")[1].split()[:3])
    assert whole > 0.1  # long enough to tell
    assert done == 0 and call < 0.3 * whole, r.stdout

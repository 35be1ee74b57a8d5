"""The launchers' size rules (wost_kernels.h), compiled for the host."""
import os
import shutil
import subprocess

import pytest

from paper_2302_11815_gb300 import build as libbuild


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """rules(expression) evaluates a C++ expression over wost_kernels.h."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    tmp = tmp_path_factory.mktemp("rules")

    def run(body):
        src, exe = str(tmp / "r.cpp"), str(tmp / "r")
        with open(src, "w") as f:
            f.write('#include <cstdio>\n#include "wost_kernels.h"\nusing namespace wost;\nint main() {' + body + "}")
        subprocess.run(["g++", "-std=c++17", "-w", "-I" + inc, "-I" + libbuild.CSRC, "-I" +
                        os.path.join(libbuild.ROOT, "include"), src, "-o", exe], check=True)
        return subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()

    return run


def test_3d_stages_spread_over_the_warps_of_the_device(rules):
    """6 warps per SM partition, 24 per SM: on 152 SMs 3,648 warps share the
    walks, on half as many SMs half as many."""
    got = rules("""
        for (int sms : {152, 76, 1, 0})
            for (unsigned long long w : {1ull, 3648ull, 3649ull, 38912ull, 1ull << 40})
                printf("%u %u\\n", spread_walks(3, w, sms), spread_walks(2, w, sms));""")
    got = [int(x) for x in got]
    assert got[1::2] == [32] * 20
    want = [min(32, max(1, -(-w // (24 * max(s, 1))))) for s in (152, 76, 1, 0) for w in (1, 3648, 3649, 38912, 1 << 40)]
    assert got[0::2] == want


def test_more_queries_than_a_grid_holds_are_asked_in_parts(rules):
    """Every query once, and every part's grid (64 threads, two queries per
    block) within 2^31 - 1 blocks."""
    got = rules("""
        for (long long n : {1ll, 1ll << 31, (1ll << 31) + 1, (1ll << 32) - 1, 1ll << 32, (1ll << 33) + 1, 1ll << 36}) {
            long long next = 0, blocks = 0;
            bool gap = false;
            in_parts(n, kWarpQueries, [&](int64_t at, int64_t m) {
                gap = gap || at != next || m < 1;
                next = at + m;
                blocks = (m + 1) / 2 > blocks ? (m + 1) / 2 : blocks;
                return cudaSuccess;
            });
            printf("%lld %lld %d\\n", next - n, blocks, (int)gap);
        }
        int calls = 0;  // an error ends it
        in_parts(1ll << 36, kWarpQueries, [&](int64_t, int64_t) { ++calls; return cudaErrorInvalidValue; });
        printf("%d\\n", calls);""")
    got = [int(x) for x in got]
    assert got[0:21:3] == [0] * 7 and got[2:21:3] == [0] * 7 and got[21] == 1
    assert all(0 < b <= 2**31 - 1 for b in got[1:21:3])

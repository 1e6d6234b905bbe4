"""When a solve runs as one launch (csrc/solve_rule.h), as plain arithmetic on the CPU: clusters that
are all resident at a time, teams with work, horizons within the limit; a launch per pass otherwise."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_03110_gb300", "csrc")

SHIM = r'''
#include "solve_rule.h"
static mhe::SolveRoom room(int teams, int sms, const int* res)
{
    mhe::SolveRoom r;
    r.teams = teams;
    r.sms = sms;
    for (int i = 0; i < mhe::kSolveSizes; ++i) r.resident[i] = res[i];
    return r;
}
extern "C" int fused(int nx, int teams, int sms, const int* res, int batch, int N)
{
    return mhe::fused_cluster(nx, room(teams, sms, res), batch, N);
}
extern "C" int resumed(int, int teams, int sms, const int* res, int batch, int N)
{
    return mhe::resumed_cluster(room(teams, sms, res), batch, N);
}
'''

# clusters of 1, 2, 4, 8, 16 CTAs resident at a time: a GPU of 152 SMs in eight groups, one CTA an SM, and two
RES1 = (152, 76, 36, 16, 4)
RES2 = (304, 152, 72, 32, 14)
TEAMS = {4: 32, 6: 32, 12: 16, 20: 8, 24: 8}


@pytest.fixture(scope="module")
def rule():
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        src, so = os.path.join(d, "s.cpp"), os.path.join(d, "s.so")
        with open(src, "w") as f:
            f.write(SHIM)
        subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
        L = ctypes.CDLL(so)
        yield lambda name, nx, res, *a: getattr(L, name)(nx, TEAMS[nx], 152, (ctypes.c_int * 5)(*res), *a)


def _limit(nx):
    return 16 if nx <= 12 else 6


@pytest.mark.parametrize("nx", sorted(TEAMS))
@pytest.mark.parametrize("res", [RES1, RES2, (152, 76, 36, 0, 0), (152, 0, 0, 0, 0)])
def test_one_launch_only_where_every_cluster_is_resident(rule, nx, res):
    taken = 0
    for batch in (1, 2, 4, 5, 8, 16, 17, 20, 36, 37, 76, 100, 152, 153, 167, 168, 400):
        for N in (1, 2, 30, 100, 128, 200, 300, 400, 600, 800, 1000, 1600, 3000, 16384):
            c = rule("fused", nx, res, batch, N)
            if c == 0:
                continue
            taken += 1
            assert c in (1, 2, 4, 8, 16)
            assert batch <= res[(1, 2, 4, 8, 16).index(c)], (batch, N, c)
            assert batch * c <= 167
            assert N <= _limit(nx) * c * TEAMS[nx]
            assert c == 1 or c * TEAMS[nx] * 10 <= N * 13   # a team has about a stage at least
    assert taken > 20


def test_measured_sides_of_the_line(rule):
    # eight instances: clusters of 16 would take two waves (nx = 12, N = 800: 0.98 ms against 0.60)
    assert rule("fused", 12, RES1, 8, 800) == 8
    assert rule("fused", 12, RES1, 4, 800) == 16
    assert rule("fused", 24, RES1, 20, 100) == 4
    # long horizons: one launch per pass
    assert rule("fused", 24, RES1, 1, 1000) == 0 and rule("fused", 20, RES1, 1, 16384) == 0
    assert rule("fused", 12, RES1, 8, 3000) == 0 and rule("fused", 12, RES1, 256, 512) == 0


@pytest.mark.parametrize("nx", sorted(TEAMS))
@pytest.mark.parametrize("res", [RES1, RES2, (152, 76, 36, 0, 0), (152, 0, 0, 0, 0), (0, 0, 0, 0, 0)])
def test_late_corrections_in_one_launch_only_where_it_cannot_cost_much(rule, nx, res):
    taken = left = 0
    for batch in (1, 2, 8, 16, 17, 36, 40, 75, 76, 100, 152, 200, 256, 304, 305, 512, 1024, 4096):
        for N in (1, 8, 31, 64, 128, 200, 300, 512, 513, 1000, 2000, 2048, 2049, 4096, 4097, 8192, 16384, 100000):
            c = rule("resumed", nx, res, batch, N)
            if c == 0:
                left += 1
                continue
            taken += 1
            size = (1, 2, 4, 8, 16).index(c)
            assert res[size] > 0
            assert N <= (32 if c >= 8 else 64) * c * TEAMS[nx]            # a single instance's share
            # one wave, unless the longest horizon asks for more CTAs an instance (then at most four)
            assert c == 1 or (batch <= res[size] and batch * c <= 167) or (c <= 4 and N > 32 * c * TEAMS[nx])
    assert left > 0 and (taken > 0) == (res[0] > 0)


def test_measured_sides_of_the_resumed_line(rule):
    # a very long horizon: the passes (one of nx = 20, N = 16384, 16 corrections: 5.2 ms, resumed 17.5)
    assert rule("resumed", 20, RES1, 1, 16384) == 0 and rule("resumed", 24, RES1, 1, 8000) == 0
    # moderate ones: clusters that fill the GPU (nx = 24, N = 1000, converged within four corrections: 0.94 ms, the passes
    # that nobody needs 1.46)
    assert rule("resumed", 24, RES1, 1, 1000) == 16 and rule("resumed", 24, RES1, 8, 1000) == 8
    assert rule("resumed", 12, RES1, 1, 6000) == 16 and rule("resumed", 20, RES1, 30, 512) == 4
    # banks and large batches: few CTAs an instance
    assert rule("resumed", 12, RES1, 256, 512) == 1 and rule("resumed", 6, RES1, 1024, 2048) == 1
    assert rule("resumed", 12, RES1, 1024, 2048) == 2 and rule("resumed", 24, RES1, 512, 2048) == 4
    assert rule("resumed", 4, RES1, 2000, 60) == 1

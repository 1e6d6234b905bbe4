"""The routes of a solve on the CPU (tests/host/engine_routes.cpp): one launch, passes, passes with the
last corrections in one launch as the shape's rules answer, wide reductions of levels with few chunks."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1510_03110_gb300", "csrc")


def test_engine_routes():
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "er")
        subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, os.path.join(ROOT, "tests", "host", "engine_routes.cpp"),
                        os.path.join(CSRC, "engine.cpp"), os.path.join(CSRC, "plan.cpp"), "-o", exe], check=True,
                       capture_output=True, text=True)
        r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout + r.stderr

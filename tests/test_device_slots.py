"""What is set once per GPU (csrc/device.h), on the CPU against a stand-in for cudaGetDevice: a
second GPU of the process gets its own call and keeps its own number, a repeated use of the
first does not, and an unknown device is never remembered."""
import os
import shutil
import subprocess
import tempfile

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_03110_gb300", "csrc")

FAKE = """
#pragma once
enum cudaError_t { cudaSuccess = 0, cudaErrorNoDevice = 100 };
extern int g_dev;
inline cudaError_t cudaGetDevice(int* d) { *d = g_dev; return g_dev < 0 ? cudaErrorNoDevice : cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
"""

MAIN = r"""
#include <stdio.h>
#include <initializer_list>
#include "device.h"
int g_dev = 0;
template <int K>
int calls()   // a launcher's once-per-GPU set-up, counted
{
    static mhe::OncePerDevice once;
    static int n = 0;
    once([] { ++n; });
    return n;
}
int number()
{
    static mhe::PerDevice per;
    return per([] { static int next = 10; return next++; });
}
int main()
{
    const int devs[] = {0, 0, 1, 0, 1, 63, 63, 64, 64, -1, -1};
    for (int d : devs) { g_dev = d; printf("%d ", calls<0>()); }
    g_dev = 0;
    printf("%d ", calls<1>());   // another kernel's set-up is its own
    for (int d : {0, 1, 0, 1, 64, 64}) { g_dev = d; printf("%d ", number()); }
}
"""


def test_every_gpu_is_set_up_once():
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        for name, text in (("cuda_runtime.h", FAKE), ("main.cpp", MAIN)):
            with open(os.path.join(d, name), "w") as f:
                f.write(text)
        exe = os.path.join(d, "t")
        subprocess.run([cxx, "-std=c++17", "-I", d, "-I", CSRC, os.path.join(d, "main.cpp"), "-o", exe], check=True,
                       capture_output=True, text=True)
        out = subprocess.run([exe], capture_output=True, text=True, timeout=60).stdout.split()
    assert out[:11] == ["1", "1", "2", "2", "2", "3", "3", "4", "5", "6", "7"]
    assert out[11] == "1"
    assert out[12:] == ["10", "11", "10", "11", "12", "13"]


def test_no_launcher_remembers_the_first_gpu_alone():
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        assert "static bool attr" not in text and "static const int most" not in text, f
        assert "static const int sms" not in text, f

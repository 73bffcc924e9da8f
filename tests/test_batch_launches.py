"""Teams of blocks count their steps in 32 bits: a launch takes no more steps than the counter of the
largest team can count, whatever number of steps a call asks for."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_08163_gb300", "csrc")

HOST = r"""
#include "lbm_internal.h"
extern "C" long long steps(long long n) { return lbmh::team_launch_steps(n); }
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("launches")
    (d / "host.cpp").write_text(HOST)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                        "-I", os.path.join(cuda, "include"), str(d / "host.cpp"), "-o", str(d / "host.so")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    fn = ctypes.CDLL(str(d / "host.so")).steps
    fn.restype, fn.argtypes = ctypes.c_longlong, [ctypes.c_longlong]
    return fn


@pytest.mark.parametrize("n", [1, 2, 1999, 2000, 2001, 7_100_000, 2 ** 31, 2 ** 40, 2 ** 62])
def test_a_launch_stays_below_the_counter(steps, n):
    m = steps(n)
    assert 1 <= m <= n and (n - m == 0 or m >= 1000)
    # resident blocks: at most 32 on an SM.  Barrier s waits for (s + 1) x parts arrivals: more than all
    # but one block's (no block passes early), and never past 2^32, where a smaller number would do
    for parts in (2, 608, 32 * 160):
        for s in (0, m // 2, m - 1):
            want = (s + 1) * parts % 2 ** 32
            assert s * parts + parts - 1 < want

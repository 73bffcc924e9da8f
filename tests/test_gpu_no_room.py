"""Allocations that fail (a stand-in for cudaMalloc that refuses some calls): a lattice whose padding does
not fit has unpadded rows, steps alike, and is tuned on a proxy with the same rows."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int from = -1, count = 0, calls = 0, seen = 0;
void refuse(int first, int n) { from = first; count = n; calls = 0; seen = 0; }
int refused(void) { return seen; }
int cudaMalloc(void **p, size_t n) {
    static int (*real)(void **, size_t);
    if (!real) real = (int (*)(void **, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
    const int k = calls++;
    if (from >= 0 && k >= from && k < from + count) {
        ++seen;
        return 2; /* cudaErrorMemoryAllocation */
    }
    return real(p, n);
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import torch
from paper_2303_08163_gb300 import inputs, lbm
shim = ctypes.CDLL(sys.argv[2])
torch.zeros(1, device="cuda")
lbm.load()
dims = (67, 40, 30)
rho, u = inputs.random_state(3, dims, seed=5, u_max=0.05)
ref = lbm.Lattice(lbm.D3Q27, dims, 0.6, 0, 0, lbm.F16S)
padded = ref.launch_info()["storage_bytes"]
assert ref.launch_info()["kernel"] == lbm.KERNEL_TMA
ref.init_fields(rho, u)
ref.step(5)
want = ref.get_populations("storage")
# the populations' allocation refused; the populations fit and what comes after them does not (with the
# numbered words and without them)
for first, n in ((0, 1), (1, 2)):
    shim.refuse(first, n)
    lat = lbm.Lattice(lbm.D3Q27, dims, 0.6, 0, 0, lbm.F16S)
    assert shim.refused() == n
    shim.refuse(-1, 0)
    info = lat.launch_info()
    assert info["kernel"] == lbm.KERNEL_GENERIC and info["storage_bytes"] < padded, info
    lat.init_fields(rho, u)
    lat.step(2)
    f = lat.get_populations("storage")
    lat.set_option(lbm.OPT_TUNE, 1)   # there is room for padding now: the proxy must not have it
    assert lat.launch_info()["kernel"] == lbm.KERNEL_GENERIC
    assert np.array_equal(lat.get_populations("storage"), f)
    lat.step(3)
    assert np.array_equal(lat.get_populations("storage"), want)
    lat.sync()
    lat.close()
# no room at all, with and without the padding
shim.refuse(0, 100)
try:
    lbm.Lattice(lbm.D3Q27, dims, 0.6, 0, 0, lbm.F16S)
    raise SystemExit("created")
except lbm.LBMError as e:
    assert e.status == lbm.ENOMEM
print("OK")
"""


def test_creation_without_room_for_padding(tmp_path):
    cc = shutil.which("gcc") or "gcc"
    src, shim = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    r = subprocess.run([cc, "-shared", "-fPIC", str(src), "-o", str(shim), "-ldl"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(shim)], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, LD_PRELOAD=str(shim)))
    assert r.returncode == 0 and "OK" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]

"""The stability search of many pairs: host memory for what goes in and out, not for the state of the search."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import resource, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import torch
from paper_2303_08163_gb300 import lbm
torch.zeros(1, device="cuda")
n = 300000
rng = np.random.default_rng(1)
nu, th = 10.0 ** rng.uniform(-3, 0, n), rng.uniform(0.05, 1.5, n)
few = lbm.vn_stability_limit(2, nu[:5000], th[:5000], nk=2, u_hi=0.9, iterations=4, tol=1e-7)
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
many = lbm.vn_stability_limit(2, nu, th, nk=2, u_hi=0.9, iterations=4, tol=1e-7)
grown = (resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before) / 1024
assert np.array_equal(many[:5000], few)
print("GROWN", grown)
"""


def test_host_memory_of_many_pairs():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    grown = float(r.stdout.split("GROWN")[1])
    # 300 000 pairs: 4.8 MB in, 2.4 MB out, a staging copy of each at most
    assert grown < 60, grown

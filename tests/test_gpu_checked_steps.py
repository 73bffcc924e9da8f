"""The bounds-checked build over the kernels of several steps and of batches (tests/checked_steps.py): no
check may fail, and the stored states equal the normal library's bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_checked_build_of_several_steps_and_batches(tmp_path):
    from paper_2303_08163_gb300 import build, lbm
    checked = build.build(checked=True)
    out = str(tmp_path / "checked.npz")
    env = dict(os.environ, LBM_LIBRARY=checked, PYTHONPATH=os.pathsep.join([HERE, ROOT, os.environ.get("PYTHONPATH", "")]))
    r = subprocess.run([sys.executable, os.path.join(HERE, "checked_steps.py"), out], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    sys.path.insert(0, HERE)
    import checked_steps
    normal = str(tmp_path / "normal.npz")
    checked_steps.run(lbm, normal)
    a, b = np.load(out), np.load(normal)
    assert sorted(a.files) == sorted(b.files) and len(a.files) == 5 * len(checked_steps.LATTICES) + 2 * len(checked_steps.BATCHES)
    for k in a.files:
        assert np.array_equal(a[k], b[k]), f"{k}: checked and normal builds differ"

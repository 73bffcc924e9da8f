"""Long FP64 runs on the paths that a program gets by default (small lattices: a cell on three lanes or on
a thread, many steps a launch; batches: clusters and teams) against the oracle: 1e-12 after the last step."""
import os

import numpy as np
import pytest

from oracle import core
from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu


def max_rel(a, b):
    return float(np.max(np.abs(a - b) / np.abs(b)))


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 1), (2, 1)])
@pytest.mark.parametrize("D,n,steps", [(2, 64, 1000), (2, 100, 1000), (3, 16, 1000), (3, 24, 300)])
def test_vortex(D, n, steps, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    dims = (n, n, 1 if D == 2 else n)
    rho, u = inputs.taylor_green_2d(n, u0=0.05) if D == 2 else inputs.taylor_green_3d(n, u0=0.05)
    core.set_threads(os.cpu_count() or 1)
    try:
        ref = core.step(D, dims, eq, bulk, 0.8, steps, core.init(D, dims, eq, rho, u))
    finally:
        core.set_threads(1)
    lat = lbm.Lattice(D - 2, dims, 0.8, eq, bulk, lbm.F64)
    lat.init_fields(rho, u)
    lat.step(steps)
    assert max_rel(lat.get_populations(), ref) <= 1e-12
    lat.close()


@pytest.mark.parametrize("dims", [[(128, 1, 1)] * 3 + [(64, 3, 1)], [(90, 81, 1), (5, 4, 1), (16, 33, 1)]])
def test_batch(dims):
    """Clusters; teams."""
    from paper_2303_08163_gb300 import lbm
    dims = np.array(dims, dtype=np.int32)
    fields = [inputs.random_state(2, tuple(int(v) for v in d), seed=3 + i, u_max=0.05) for i, d in enumerate(dims)]
    tau = np.linspace(0.6, 0.9, len(dims))
    b = lbm.Batch(lbm.D2Q9, dims, tau, lbm.ENTROPIC, 1)
    b.init_fields(np.concatenate([f[0] for f in fields]), np.concatenate([f[1].reshape(-1) for f in fields]))
    b.step(1000)
    f = b.get_populations()
    for k, d in enumerate(dims):
        d3 = tuple(int(v) for v in d)
        ref = core.step(2, d3, 0, 1, float(tau[k]), 1000, core.init(2, d3, 0, *fields[k]))
        got = f[9 * b.cell_start[k]:9 * b.cell_start[k + 1]].reshape(9, -1)
        assert max_rel(got, ref) <= 1e-12
    b.sync()
    b.close()

"""Teams of blocks (few or uneven instances) against whole instances per block."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = {
    # one block a lattice; several; a large one beside tiny ones; more lattices than threads cover at once
    "flat": (2, [(128, 1, 1)] * 5 + [(64, 1, 1)]),
    "even": (2, [(40, 37, 1)] * 7),
    "uneven": (2, [(250, 200, 1), (1, 1, 1), (16, 3, 1), (2, 2, 1), (129, 1, 1)]),
    "one": (2, [(301, 77, 1)]),
    "many": (2, [(12 + k % 60, 9 + k % 41, 1) for k in range(220)]),
    "3d": (3, [(20, 12, 9), (3, 2, 1), (8, 8, 8), (1, 5, 4)]),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("eq,bulk", [(0, 1), (1, 0), (2, 0)])
def test_teams_match_whole_instances(name, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    D, dims = CASES[name]
    dims = np.array(dims, dtype=np.int32)
    n = len(dims)
    rng = np.random.default_rng(n + eq)
    tau = 0.5 + rng.uniform(0.05, 0.5, n)
    kvec = rng.integers(0, 3, (n, 3)).astype(np.int32)
    kvec[:, 2] *= D == 3
    fields = [inputs.random_state(D, tuple(int(v) for v in d), seed=60 + i, u_max=0.1) for i, d in enumerate(dims)]
    rho = np.concatenate([f[0] for f in fields])
    u = np.concatenate([f[1].reshape(-1) for f in fields])
    out = []
    for whole in (False, True):
        b = lbm.Batch(lbm.D2Q9 if D == 2 else lbm.D3Q27, dims, tau, eq, bulk)
        if whole:
            b.set_launch_shape(64, min(n, 3))
        b.init_fields(rho, u)
        b.set_probe(kvec, 3 if eq else 1)
        for steps in (5, 1, 8):
            b.step(steps)
        out.append((b.get_populations(), b.probe_series(), b.status(), b.info()["step"]))
        b.sync()
        b.close()
    (f0, s0, st0, t0), (f1, s1, st1, t1) = out
    assert t0 == t1 == 14 and np.array_equal(st0, st1) and not st0.any()
    assert np.max(np.abs(f0 - f1)) <= 1e-14  # the two kernels may contract differently
    cells = dims.prod(axis=1)[:, None, None]
    assert s0.shape == s1.shape and np.all(np.abs(s0 - s1) <= 1e-14 * cells)

"""FP64 cells on three lanes of a warp (small lattices and batches) against one cell per thread."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

STEPS = (2, 1, 9)
# 12 steps of some 20 roundings of values below 1/2, which may differ in order
TOL = sum(STEPS) * 20 * 2.0 ** -54

# one cell; partial groups and warps; neighbours that coincide; one block more than full blocks;
# the largest lattice of the rule on 152 SMs (6080 cells) and the next one
DIMS = [(2, (1, 1, 1)), (2, (3, 1, 1)), (2, (1, 11, 1)), (2, (2, 2, 1)), (2, (64, 64, 1)), (2, (41, 37, 1)), (2, (80, 76, 1)),
        (2, (6081, 1, 1)), (3, (1, 1, 1)), (3, (2, 3, 1)), (3, (1, 2, 31)), (3, (16, 16, 16)), (3, (19, 20, 16)), (3, (7, 11, 13))]


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("D,dims", DIMS)
def test_lanes_match_one_cell_per_thread(D, dims, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=90 + dims[0], rho_range=(0.9, 1.1), u_max=0.1)
    lats = [lbm.Lattice(D - 2, dims, 0.6, eq, bulk, 0) for _ in range(2)]
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 64)
    for lat in lats:
        lat.init_fields(rho, u)
    for n in STEPS:
        for lat in lats:
            lat.step(n)
    a, b = (lat.get_populations() for lat in lats)
    assert np.max(np.abs(a - b)) <= TOL
    for lat in lats:
        lat.sync()
        lat.close()


# full and partial blocks, a block an SM at most (152 blocks), one more
BATCHES = [(2, [(128, 1, 1)] * 28), (2, [(40, 1, 1), (1, 1, 1), (41, 1, 1), (9, 11, 1)]), (2, [(5, 8, 1)] * 152), (2, [(5, 8, 1)] * 153),
           (3, [(16, 9, 1), (1, 1, 1), (4, 5, 6)])]


@pytest.mark.parametrize("eq,bulk", [(0, 1), (1, 0), (2, 1)])
@pytest.mark.parametrize("D,dims", BATCHES)
def test_lanes_of_a_batch(D, dims, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    dims = np.array(dims, dtype=np.int32)
    n = len(dims)
    rng = np.random.default_rng(n)
    tau = 0.5 + rng.uniform(0.05, 0.5, n)
    kvec = rng.integers(0, 3, (n, 3)).astype(np.int32)
    kvec[:, 2] *= D == 3
    fields = [inputs.random_state(D, tuple(int(v) for v in d), seed=20 + i, u_max=0.1) for i, d in enumerate(dims)]
    rho = np.concatenate([f[0] for f in fields])
    u = np.concatenate([f[1].reshape(-1) for f in fields])
    out = []
    for whole in (False, True):
        b = lbm.Batch(lbm.D2Q9 if D == 2 else lbm.D3Q27, dims, tau, eq, bulk)
        if whole:
            b.set_launch_shape(64, min(n, 3))
        b.init_fields(rho, u)
        b.set_probe(kvec, 2)
        for steps in STEPS:
            b.step(steps)
        out.append((b.get_populations(), b.probe_series(), b.status()))
        b.close()
    (f0, s0, st0), (f1, s1, st1) = out
    assert np.array_equal(st0, st1) and not st0.any()
    assert np.max(np.abs(f0 - f1)) <= TOL
    cells = dims.prod(axis=1)[:, None, None]
    assert s0.shape == s1.shape and np.all(np.abs(s0 - s1) <= 9 * TOL * cells)

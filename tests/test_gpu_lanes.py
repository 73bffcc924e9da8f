"""FP64 cells on three lanes of a warp (small lattices) against one cell per thread."""
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

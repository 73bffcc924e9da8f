"""Several steps of a small lattice in one launch, populations numbered by step, against one launch
per step of the one-cell kernel."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

# on 152 SMs: the largest lattice of each rule and the next one; one, two and more blocks an SM, two and
# three rounds; padded and ragged rows; coinciding neighbours
CASES = [(2, (512, 608, 1), 1), (2, (512, 609, 1), 1), (2, (320, 608, 1), 2), (2, (320, 609, 1), 2), (2, (256, 608, 1), 0),
         (2, (256, 609, 1), 0), (2, (300, 301, 1), 2), (2, (333, 512, 1), 1), (2, (1, 700, 1), 2), (2, (2, 1, 1), 1),
         (3, (60, 62, 62), 2), (3, (62, 62, 61), 2), (3, (48, 48, 50), 2), (3, (32, 32, 114), 1), (3, (29, 32, 76), 1),
         (3, (32, 32, 114), 0), (3, (32, 32, 115), 0), (3, (32, 38, 64), 0), (3, (32, 38, 65), 0), (3, (1, 2, 3), 2), (3, (31, 40, 31), 2)]


def pair(lbm, D, dims, prec, eq=0, bulk=1):
    rho, u = inputs.random_state(D, dims, seed=sum(dims), rho_range=(0.9, 1.1), u_max=0.05)
    lats = [lbm.Lattice(D - 2, dims, 0.7, eq, bulk, prec) for _ in range(2)]
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 128)
    for lat in lats:
        lat.init_fields(rho, u)
    return lats


@pytest.mark.parametrize("D,dims,prec", CASES)
def test_sizes_of_the_rule(D, dims, prec):
    from paper_2303_08163_gb300 import lbm
    lats = pair(lbm, D, dims, prec)
    for n in (3, 2, 20):
        for lat in lats:
            lat.step(n)
        a, b = (lat.get_populations("storage") for lat in lats)
        if prec == 0:  # 25 steps of some 20 roundings of values below 1/2, which may differ
            assert np.max(np.abs(a - b)) <= 25 * 20 * 2.0 ** -54
        else:
            assert np.array_equal(a, b)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("D,dims,prec,eq", [(2, (16, 9, 1), 2, 0), (2, (16, 9, 1), 1, 1), (3, (6, 5, 4), 2, 2)])
def test_step_numbers_go_on(D, dims, prec, eq):
    """More steps than a 16-bit number counts, over many launches."""
    from paper_2303_08163_gb300 import lbm
    lats = pair(lbm, D, dims, prec, eq)
    for n in (65530, 2, 2, 2, 3, 5, 4001):
        for lat in lats:
            lat.step(n)
        assert np.array_equal(*(lat.get_populations("storage") for lat in lats))
    for lat in lats:
        lat.close()

"""The shared memory limit of a step kernel belongs to the kernel function, which lattices of one kind
share: creating a second lattice must not take from the first what its launch shape needs."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,dims,prec,shape", [(2, (256, 96, 1), 1, (2, 128, 3, 4, 256, 4096)), (3, (64, 32, 20), 2, (2, 128, 4, 4, 64, 1024)),
                                               (2, (512, 40, 1), 2, (2, 256, 8, 1, 512, 2048))])
def test_a_second_lattice_leaves_the_first_its_stages(D, dims, prec, shape):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=3, u_max=0.05)
    first = lbm.Lattice(D - 2, dims, 0.6, lbm.ENTROPIC, 0, prec)
    first.set_launch_shape(*shape)
    first.init_fields(rho, u)
    first.step(1)
    # the smallest shape of the same kernel, then one with the default shape
    small = lbm.Lattice(D - 2, dims, 0.6, lbm.ENTROPIC, 0, prec)
    small.set_launch_shape(2, shape[1], 2, *shape[3:])
    second = lbm.Lattice(D - 2, dims, 0.6, lbm.ENTROPIC, 0, prec)
    for lat in (small, second):
        lat.init_fields(rho, u)
        lat.step(1)
    for n in (1, 3):
        for lat in (first, small, second):
            lat.step(n)
    got = [lat.get_populations("storage") for lat in (first, small, second)]
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    for lat in (first, small, second):
        lat.sync()
        lat.close()

"""Several steps a launch with the TMA row kernel where its order of jobs has its edges, against the
one-cell kernel launched step by step: few positions, strips, odd rows, and the packed collision.  Small
lattices get a launch shape, without which they would take the kernels for small lattices."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

# (D, dims, precision, shape or None): one, two, three positions along the sweep and across it; a
# position in several jobs; short last groups; whole rows and segments; padded rows of odd and even length
FEW = [
    (2, (64, 1, 1), 0, (2, 64, 2, 1, 64, 1024)), (2, (64, 2, 1), 1, (2, 128, 3, 1, 64, 1024)), (2, (48, 3, 1), 2, (2, 64, 2, 1, 48, 1024)),
    (2, (48, 5, 1), 2, (2, 64, 2, 4, 48, 1024)), (2, (256, 2, 1), 1, (2, 128, 2, 1, 64, 1024)), (2, (256, 1, 1), 2, (2, 128, 2, 1, 72, 1024)),
    (3, (16, 9, 1), 1, (2, 64, 2, 2, 16, 1024)), (3, (16, 5, 2), 2, (2, 64, 2, 5, 16, 1024)), (3, (16, 1, 3), 0, (2, 32, 2, 1, 16, 1024)),
    (3, (48, 2, 7), 2, (2, 64, 4, 1, 48, 1024)), (3, (48, 40, 3), 2, (2, 128, 2, 7, 48, 1024)), (3, (96, 3, 2), 1, (2, 128, 2, 1, 48, 1024)),
    (3, (67, 3, 1), 2, (2, 128, 2, 2, 67, 1024)), (3, (33, 2, 2), 1, (2, 128, 2, 1, 33, 1024)), (2, (131, 3, 1), 2, (2, 128, 2, 2, 131, 1024)),
    (2, (509, 2, 1), 1, (2, 128, 2, 1, 509, 4096)), (2, (66, 1, 1), 2, (2, 64, 2, 1, 66, 1024)),
    # by default: one position, and odd rows beyond the small lattices
    (3, (512, 512, 1), 2, None), (3, (512, 300, 2), 1, None), (3, (301, 40, 30), 2, None), (3, (203, 45, 40), 1, None), (2, (2047, 300, 1), 1, None),
    (2, (1001, 400, 1), 2, None),
]


def pair(lbm, D, dims, prec, shape, eq=0, bulk=1):
    lats = [lbm.Lattice(D - 2, dims, 0.7, eq, bulk, prec) for _ in range(2)]
    if shape:
        lats[0].set_launch_shape(*shape)
    assert lats[0].launch_info()["kernel"] == lbm.KERNEL_TMA
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 128)
    return lats


@pytest.mark.parametrize("D,dims,prec,shape", FEW)
def test_few_positions(D, dims, prec, shape):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=50 + dims[1], rho_range=(0.9, 1.1), u_max=0.05)
    lats = pair(lbm, D, dims, prec, shape)
    for lat in lats:
        lat.init_fields(rho, u)
    for n in (2, 3, 1, 40, 17):
        for lat in lats:
            lat.step(n)
        assert np.array_equal(*(lat.get_populations("storage") for lat in lats)), n
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("D,dims,prec", [(3, (256, 40, 24), 2), (3, (128, 40, 24), 1), (3, (131, 40, 24), 2), (3, (133, 40, 24), 1),
                                         (2, (512, 1000, 1), 2), (2, (512, 1000, 1), 1), (2, (511, 1000, 1), 2), (2, (1031, 700, 1), 1)])
def test_packed_collisions(D, dims, prec, eq, bulk):
    """Two cells a thread, even and odd steps within a launch."""
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=80 + eq, u_max=0.15)
    lats = pair(lbm, D, dims, prec, None, eq, bulk)
    for lat in lats:
        lat.init_fields(rho, u)
    for n in (2, 3, 2):
        for lat in lats:
            lat.step(n)
        assert np.array_equal(*(lat.get_populations("storage") for lat in lats)), n
    for lat in lats:
        lat.close()


# on 152 SMs swept three steps at a time in 3, 5 and 10 strips; numbers of steps that are no multiple of it
@pytest.mark.parametrize("dims,prec", [((256, 256, 256), 1), ((512, 512, 512), 2), ((512, 512, 500), 1)])
def test_strips(dims, prec):
    import torch
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state_torch(3, dims, seed=6, u_max=0.05)
    lats = pair(lbm, 3, dims, prec, None, bulk=0)
    st = {1: torch.float32, 2: torch.float16}[prec]
    for lat in lats:
        lat.init_fields(rho, u, dtype=np.float32)
    for n in (7, 4):
        for lat in lats:
            lat.step(n)
        a, b = (lat.get_populations("storage", out=torch.empty((lat.Q, lat.ncell), dtype=st, device="cuda")) for lat in lats)
        assert torch.equal(a, b), n
        del a, b
    for lat in lats:
        lat.sync()
        lat.close()

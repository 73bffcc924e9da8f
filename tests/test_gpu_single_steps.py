"""Steps launched one by one with the TMA row kernel (one service warp that stores and refills),
with and without diagnostics, against the one-cell kernel on the same stored values."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

# (D, dims, precision, shape or None): one job, fewer jobs than stages, as many, one more, many a block;
# rows, segments with a short last one, padded rows of odd and even length; the default shapes
CASES = [
    (2, (64, 1, 1), 1, (2, 64, 3, 1, 64, 1024)), (2, (64, 2, 1), 0, (2, 32, 4, 1, 64, 1024)), (2, (64, 700, 1), 2, (2, 64, 8, 1, 64, 1024)),
    (2, (96, 1217, 1), 1, (2, 128, 2, 1, 96, 1024)), (2, (200, 330, 1), 1, (2, 96, 3, 1, 72, 1024)), (2, (520, 77, 1), 2, (2, 512, 2, 1, 264, 1024)),
    (3, (8, 1, 1), 2, (2, 32, 2, 1, 8, 1024)), (3, (16, 3, 2), 2, (2, 64, 3, 2, 16, 1024)), (3, (48, 20, 19), 1, (2, 128, 2, 3, 48, 1024)),
    (3, (96, 64, 20), 2, (2, 128, 2, 1, 48, 1024)), (3, (24, 40, 30), 0, (2, 128, 2, 5, 24, 1024)),
    (3, (67, 33, 29), 2, None), (3, (33, 40, 21), 1, None), (2, (509, 381, 1), 1, None), (2, (130, 411, 1), 2, None),
    (2, (1536, 1501, 1), 1, None), (2, (1000, 1100, 1), 0, None),
]


@pytest.mark.parametrize("D,dims,prec,shape", CASES)
@pytest.mark.parametrize("eq,bulk", [(0, 1), (1, 0)])
def test_single_steps(D, dims, prec, shape, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=30 + dims[1], rho_range=(0.9, 1.1), u_max=0.05)
    lats = [lbm.Lattice(D - 2, dims, 0.7, eq, bulk, prec) for _ in range(3)]
    if shape:
        for lat in lats[:2]:
            lat.set_launch_shape(*shape)
    lats[2].set_launch_shape(lbm.KERNEL_GENERIC, 128)
    for lat in lats:
        assert lat is lats[2] or lat.launch_info()["kernel"] == lbm.KERNEL_TMA
        lat.init_fields(rho, u)
    lats[1].set_option(lbm.OPT_DIAG_EVERY, 1)
    for _ in range(5):
        for lat in lats:
            lat.step(1)
    got = [lat.get_populations("storage") for lat in lats]
    assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[2])
    d = lats[1].diag_history()
    assert [x["step"] for x in d] == list(range(5)) and all(x["nonfinite"] == 0 for x in d)
    # mass is conserved: FP32 partial sums of at most 2^13 deviations below 0.2, and the storage's rounding
    n, eps = lats[0].ncell, (2.0 ** -50, 2.0 ** -22, 2.0 ** -11)[prec]
    assert all(abs(x["mass"] - rho.sum()) <= n * eps for x in d)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("dims", [(300, 500, 1), (512, 400, 1), (640, 260, 1)])
def test_few_fp64_steps(dims):
    """Numbers of FP64 steps on both sides of the rule, at both parities."""
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(2, dims, seed=3, u_max=0.1)
    lats = [lbm.Lattice(lbm.D2Q9, dims, 0.6, 0, 1, lbm.F64) for _ in range(2)]
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 128)
    for lat in lats:
        lat.init_fields(rho, u)
    for n in (2, 3, 4, 5, 6, 1, 4, 5):
        for lat in lats:
            lat.step(n)
        assert np.array_equal(*(lat.get_populations("storage") for lat in lats)), n
    for lat in lats:
        lat.close()

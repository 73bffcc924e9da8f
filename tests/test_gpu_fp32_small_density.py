"""FP32 densities down to the edge of the normal numbers and a little below it."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 1), (2, 0)])
@pytest.mark.parametrize("D,dims", [(2, (64, 40, 1)), (2, (63, 41, 1)), (3, (24, 10, 6))])
def test_densities_at_the_edge(D, dims, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=4, rho_range=(0.8, 1.2), u_max=0.1)

    def run(scale, calls, shape):
        lat = lbm.Lattice(D - 2, dims, 0.6, eq, bulk, lbm.F32, rho0=scale)
        if shape:
            lat.set_launch_shape(*shape)
        lat.init_fields(rho * scale, u)
        for n in calls:
            lat.step(n)
        f = lat.get_populations() / scale
        lat.close()
        return f

    for calls in ((3,), (1, 1, 1)):
        for shape in (None, (lbm.KERNEL_GENERIC, 64)):
            want = run(1.0, calls, shape)
            for scale in (1.2e-38, 1.3e-37):
                # 3 steps, each of the populations' roundings to multiples of 2^-149 and FP32's own
                tol = 3 * 3 ** D * (2.0 ** -149 / scale + 2.0 ** -24)
                assert np.max(np.abs(run(scale, calls, shape) - want)) <= tol, (scale, calls, shape)

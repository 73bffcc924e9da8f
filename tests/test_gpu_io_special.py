"""Infinite and undefined populations through FP32 import and export: as the FP64 sum has them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W1 = np.array([1 / 6, 2 / 3, 1 / 6])


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("D,dims", [(2, (64, 3, 1)), (2, (7, 5, 1)), (3, (66, 2, 3)), (3, (67, 2, 2))])
def test_infinities_pass_through(D, dims, prec):
    from paper_2303_08163_gb300 import lbm
    lat = lbm.Lattice(D - 2, dims, 0.6, 0, 0, prec, rho0=1.1)
    w = (np.multiply.outer(W1, W1) if D == 2 else np.multiply.outer(W1, np.multiply.outer(W1, W1))).reshape(-1, 1)
    rng = np.random.default_rng(dims[0])
    st = rng.uniform(-0.1, 0.1, (lat.Q, lat.ncell)).astype(lbm.STORAGE_NUMPY[prec])
    at = rng.permutation(st.size)[:60]
    st.flat[at[:20]], st.flat[at[20:40]], st.flat[at[40:]] = np.inf, -np.inf, np.nan
    for step in (0, 1):
        lat.set_step_count(step)
        lat.set_populations(st, "storage")
        got = lat.get_populations(np.float32)
        want = (st.astype(np.float64) + w * 1.1).astype(np.float32)
        for special in (np.isposinf, np.isneginf, np.isnan):
            assert np.array_equal(special(got), special(want))
        fin = np.isfinite(want)
        assert np.all(np.abs(got[fin] - want[fin]) <= np.spacing(np.abs(want[fin])))
        lat.set_populations(want, np.float32)
        back = lat.get_populations("storage")
        for special in (np.isposinf, np.isneginf, np.isnan):
            assert np.array_equal(special(back), special(want))
    lat.close()

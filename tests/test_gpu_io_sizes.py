"""Field and population transfers on both sides of the sizes where binary16 cells go in pairs, on padded
and unpadded rows, at both parities, against NumPy on the stored values."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

W1 = np.array([1 / 6, 2 / 3, 1 / 6])

# (D, dims, precision): just below and above 2^17 and 2^21 cells; even, odd and padded rows
CASES = [(2, (256, 511, 1), 2), (2, (256, 512, 1), 2), (2, (257, 511, 1), 2), (2, (250, 530, 1), 2), (3, (67, 45, 44), 2), (3, (66, 45, 45), 2),
         (2, (2048, 1023, 1), 2), (2, (2050, 1024, 1), 2), (2, (2049, 1025, 1), 2), (2, (509, 381, 1), 1), (3, (131, 9, 7), 1), (3, (7, 5, 3), 1),
         (3, (33, 20, 11), 0)]


@pytest.mark.parametrize("D,dims,prec", CASES)
def test_transfers(D, dims, prec):
    from paper_2303_08163_gb300 import lbm
    rho0 = 1.1
    rho, u = inputs.random_state(D, dims, seed=dims[0], rho_range=(1.0, 1.2), u_max=0.1)
    lat = lbm.Lattice(D - 2, dims, 0.6, 0, 0, prec, rho0=rho0)
    ref = lbm.Lattice(D - 2, dims, 0.6, 0, 0, lbm.F64, rho0=rho0)
    st_t = lbm.STORAGE_NUMPY[prec]
    wr = (np.multiply.outer(W1, W1) if D == 2 else np.multiply.outer(W1, np.multiply.outer(W1, W1))).reshape(-1, 1) * rho0
    # initialisation: FP64's to the rounding of the FP32 terms (some ten operations on values below 1) and the storage
    lat.init_fields(rho, u)
    ref.init_fields(rho, u)
    eps = (0, 2.0 ** -21, 2.0 ** -11)[prec]
    want = ref.get_populations("storage")
    got = lat.get_populations("storage").astype(np.float64)
    assert np.all(np.abs(got - want) <= eps * (np.abs(want) + 2.0 ** -3) + 1e-16)
    ref.close()
    # an asymmetric state, written and read in every type
    rng = np.random.default_rng(dims[1])
    st = rng.uniform(-0.05, 0.05, (lat.Q, lat.ncell)).astype(st_t)
    for step in (0, 1):
        lat.set_step_count(step)
        lat.set_populations(st, "storage")
        assert np.array_equal(lat.get_populations("storage"), st)
        for dt in (np.float32, np.float64):
            f = lat.get_populations(dt)
            exact = st.astype(np.float64) + wr
            assert np.all(np.abs(f - exact.astype(dt)) <= np.spacing(np.abs(exact).astype(dt)))
            lat.set_populations(np.zeros_like(f), dt)
            lat.set_populations(f, dt)
            back = (f.astype(np.float64) - wr).astype(np.float64 if prec == 0 else np.float32).astype(st_t)
            assert np.all(np.abs(lat.get_populations("storage").astype(np.float64) - back) <= np.spacing(np.abs(back)).astype(np.float64))
            lat.set_populations(st, "storage")
            r, v = lat.moments(dt)
            s64 = st.astype(np.float64)
            assert np.allclose(r, rho0 + s64.sum(0), rtol=0, atol=1e-12 if prec == 0 and dt == np.float64 else 64 * 2 ** -24)
    # a step on the padded state does not see the padding
    gen = lbm.Lattice(D - 2, dims, 0.6, 0, 0, prec, rho0=rho0)
    gen.set_launch_shape(lbm.KERNEL_GENERIC, 128)
    for x in (lat, gen):
        x.set_step_count(0)
        x.init_fields(rho, u)
        x.step(3)
    assert np.array_equal(lat.get_populations("storage"), gen.get_populations("storage"))
    lat.close()
    gen.close()

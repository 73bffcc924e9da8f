"""Population import and export in FP32 (sums carried in FP32 pairs) and the two-cell forms of the
field kernels, at both parities, against NumPy on the stored values."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

W1 = np.array([1 / 6, 2 / 3, 1 / 6])


def weights(D):
    w = np.multiply.outer(W1, W1) if D == 2 else np.multiply.outer(W1, np.multiply.outer(W1, W1))
    return w.reshape(-1, 1)


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("D,dims", [(3, (66, 5, 3)), (3, (67, 4, 3)), (3, (1, 2, 3)), (2, (64, 3, 1)), (2, (131, 2, 1)),
                                    (2, (7, 5, 1)), (2, (2, 1, 1))])
def test_fp32_populations_round_like_fp64_sums(D, dims, prec):
    from paper_2303_08163_gb300 import lbm
    rho0 = 1.1
    rho, u = inputs.random_state(D, dims, seed=5 + dims[0], rho_range=(1.0, 1.2), u_max=0.1)
    lat = lbm.Lattice(D - 2, dims, 0.6, 0, 0, prec, rho0=rho0)
    lat.init_fields(rho, u)
    wr = weights(D) * rho0
    for n in (0, 1):
        lat.step(n)
        st = lat.get_populations("storage")
        got = lat.get_populations(np.float32)
        want = (st.astype(np.float64) + wr).astype(np.float32)
        assert np.all(np.abs(got - want) <= np.spacing(np.abs(want)))
        # writing them back: the FP64 difference rounded to FP32, then to the storage type
        lat.set_populations(got, np.float32)
        back = lat.get_populations("storage")
        d = (got.astype(np.float64) - wr).astype(np.float32 if prec else np.float64)
        if prec == 2:
            d = d.astype(np.float16)
        assert np.all(np.abs(back.astype(np.float64) - d) <= np.spacing(np.abs(d)).astype(np.float64))
        # moments of what is stored now
        r, v = lat.moments()
        f = back.astype(np.float64)
        assert np.allclose(r, rho0 + f.sum(0), rtol=0, atol=1e-12 if prec == 0 else 64 * 2 ** -24)
    lat.close()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("D,dims", [(3, (66, 5, 3)), (2, (64, 3, 1))])
def test_outputs_that_start_between_pairs(D, dims, dtype):
    """Device outputs aligned to one value only, against aligned ones: the same bits."""
    import torch
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=8, u_max=0.1)
    lat = lbm.Lattice(D - 2, dims, 0.6, 0, 0, 2)
    lat.init_fields(rho, u)
    td = torch.float32 if dtype == np.float32 else torch.float64
    n = lat.ncell

    def take(off):
        r = torch.zeros(n + 4, dtype=td, device="cuda")[off:off + n]
        v = torch.zeros(D * n + 4, dtype=td, device="cuda")[off:off + D * n].view(D, n)
        f = torch.zeros(lat.Q * n + 4, dtype=td, device="cuda")[off:off + lat.Q * n].view(lat.Q, n)
        lat.moments(dtype, out=(r, v))
        lat.get_populations(dtype, out=f)
        torch.cuda.synchronize()
        return r, v, f

    for steps in (0, 1):
        lat.step(steps)
        for a, b in zip(take(0), take(1)):
            assert torch.equal(a, b)
    lat.close()

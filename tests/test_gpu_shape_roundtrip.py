"""A launch shape that one lattice reports can be set on another of its kind and size, ragged rows
included, and stores the same bits."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,dims,prec", [(2, (509, 381, 1), 1), (3, (67, 20, 11), 2), (2, (131, 97, 1), 2), (2, (256, 300, 1), 1),
                                         (3, (48, 20, 19), 2), (2, (13, 8, 1), 1), (2, (64, 64, 1), 0)])
@pytest.mark.parametrize("tune", [0, 1])
def test_reported_shape_can_be_set(D, dims, prec, tune):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=11, u_max=0.05)
    lats = [lbm.Lattice(D - 2, dims, 0.6, lbm.ENTROPIC, 0, prec) for _ in range(2)]
    lats[0].init_fields(rho, u)
    if tune:
        lats[0].set_option(lbm.OPT_TUNE, 1)
    i = lats[0].launch_info()
    cap = i["smem_bytes"] // (lats[0].Q * i["stages"]) if i["kernel"] == lbm.KERNEL_TMA else 0
    lats[1].set_launch_shape(i["kernel"], i["threads"], i["stages"], i["rows"], i["seg"], cap)
    j = lats[1].launch_info()
    assert all(i[k] == j[k] for k in ("kernel", "threads", "stages", "rows", "seg", "smem_bytes"))
    lats[1].init_fields(rho, u)
    for n in (1, 4):
        for lat in lats:
            lat.step(n)
        assert np.array_equal(*(lat.get_populations("storage") for lat in lats))
    if i["kernel"] == lbm.KERNEL_TMA and dims[0] % 8:
        with pytest.raises(lbm.LBMError) as e:  # padded rows go whole
            lats[1].set_launch_shape(i["kernel"], i["threads"], i["stages"], 1, 16, cap)
        assert e.value.status == lbm.EINVAL
    for lat in lats:
        lat.close()

"""Lattices whose rows are no multiple of 16 bytes: padded rows through the TMA row kernel
against the one-cell kernel on the same stored values."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

# (D, dims, precision): odd and even row lengths, one-row jobs and several rows, y wrap,
# the longest padded rows of each buffer size
CASES = [
    (3, (67, 5, 4), 2), (3, (66, 7, 3), 2), (3, (250, 9, 5), 2), (3, (65, 1, 2), 2), (3, (1027, 3, 2), 2),
    (3, (2047, 2, 2), 2), (2, (65, 33, 1), 2), (2, (4095, 3, 1), 2), (2, (1022, 5, 1), 2),
    (3, (33, 6, 5), 1), (3, (1023, 3, 2), 1), (2, (509, 7, 1), 1), (2, (2047, 4, 1), 1), (2, (35, 1, 1), 1),
]


@pytest.mark.parametrize("D,dims,prec", CASES)
@pytest.mark.parametrize("eq,bulk", [(0, 1), (1, 0)])
def test_padded_rows_match_one_cell_kernel(D, dims, prec, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=40 + dims[0], u_max=0.1)
    lats = []
    for generic in (False, True):
        lat = lbm.Lattice(D - 2, dims, 0.6, eq, bulk, prec)
        assert lat.launch_info()["kernel"] == lbm.KERNEL_TMA
        with pytest.raises(lbm.LBMError):
            lat.set_option(lbm.OPT_KERNEL, 2)  # asking for the TMA kernel needs 16-byte rows
        if generic:
            lat.set_launch_shape(lbm.KERNEL_GENERIC, 128)
        lat.set_option(lbm.OPT_DIAG_EVERY, 2)
        lat.init_fields(rho, u)
        lats.append(lat)
    for n in (1, 1, 3):
        for lat in lats:
            lat.step(n)
        assert np.array_equal(lats[0].get_populations("storage"), lats[1].get_populations("storage"))
    for a, b in zip(lats[0].moments(), lats[1].moments()):
        assert np.array_equal(a, b)
    # per-cell sums in another order: FP32 partials over at most 128 cells
    for a, b in zip(lats[0].diag_history(), lats[1].diag_history()):
        assert abs(a["mass"] - b["mass"]) <= 2 * 2 ** -24 * 155 * abs(b["mass"])
        assert a["max_u"] == b["max_u"] and a["nonfinite"] == b["nonfinite"] == 0
    # a checkpoint of the padded lattice restores into it, at both parities
    for n in (0, 1):
        lats[0].step(n)
        f = lats[0].get_populations("storage")
        lats[0].set_populations(f, "storage")
        assert np.array_equal(lats[0].get_populations("storage"), f)
    for lat in lats:
        lat.close()

"""A team's wait that runs out is reported, also when the batch has another launch shape by then."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("other_shape", [False, True])
def test_expired_wait_is_reported(other_shape, monkeypatch):
    """A wait limit of a nanosecond: the blocks of one large instance, which no number of SMs shares out
    evenly, differ by more than a poll loop, give up and return."""
    from paper_2303_08163_gb300 import lbm
    dims = np.array([(2000, 2011, 1), (3, 2, 1)], dtype=np.int32)
    total = int(dims.prod(axis=1).sum())
    b = lbm.Batch(lbm.D2Q9, dims, np.array([0.7, 0.8]))
    b.init_fields(np.ones(total), np.full(2 * total, 0.01))
    monkeypatch.setenv("LBM_WAIT_TIMEOUT_NS", "1")
    b.step(20)
    monkeypatch.delenv("LBM_WAIT_TIMEOUT_NS")
    if other_shape:
        b.set_launch_shape(128, 2)
    with pytest.raises(lbm.LBMError) as e:
        b.sync()
    assert e.value.status == lbm.ETIMEOUT
    with pytest.raises(lbm.LBMError) as e:
        b.step(1)
    assert e.value.status == lbm.ESTATE
    b.close()

"""A call of more steps than one launch of teams takes, against whole instances per block."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_teams_over_several_launches():
    from paper_2303_08163_gb300 import lbm
    dims = np.array([(61, 40, 1), (3, 2, 1), (40, 50, 1)], dtype=np.int32)  # two uneven teams, one block
    fields = [inputs.random_state(2, tuple(int(v) for v in d), seed=7 + i, u_max=0.05) for i, d in enumerate(dims)]
    rho = np.concatenate([f[0] for f in fields])
    u = np.concatenate([f[1].reshape(-1) for f in fields])
    out = []
    for whole in (False, True):
        b = lbm.Batch(lbm.D2Q9, dims, np.array([0.6, 0.9, 0.7]), lbm.ENTROPIC, 1)
        if whole:
            b.set_launch_shape(128, 3)
        b.init_fields(rho, u)
        b.set_probe(np.array([(1, 0, 0)] * 3, dtype=np.int32), 7)
        b.step(4321)  # three launches of teams
        out.append((b.get_populations(), b.probe_series(), b.info()["step"]))
        b.sync()
        b.close()
    (f0, s0, t0), (f1, s1, t1) = out
    assert t0 == t1 == 4321 and s0.shape == s1.shape == (3, 618, 4)
    # the waves have died out: what is left are roundings of 4321 steps of some 20 operations
    tol = 4321 * 20 * 2.0 ** -54
    assert np.max(np.abs(f0 - f1)) <= tol
    assert np.all(np.abs(s0 - s1) <= 9 * tol * dims.prod(axis=1)[:, None, None])

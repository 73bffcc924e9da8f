"""FP64 states do not depend on how steps are grouped, on diagnostics or on the kernel: every kernel
stores the same bits (a cell on a thread, a cell on three lanes; single and several steps; batches of
whole instances, teams and clusters)."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

EQS = [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0), (2, 1)]


@pytest.mark.parametrize("eq,bulk", EQS)
@pytest.mark.parametrize("D,dims", [(2, (64, 64, 1)), (2, (41, 37, 1)), (2, (160, 150, 1)), (2, (512, 400, 1)), (3, (16, 16, 16)),
                                    (3, (7, 11, 13)), (3, (30, 31, 33)), (3, (48, 48, 50)), (3, (64, 50, 60))])
def test_lattice(D, dims, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=1 + dims[0], rho_range=(0.9, 1.1), u_max=0.1)
    got = {}
    for name, calls, diag, shape in (("several", (12,), 0, None), ("split", (7, 5), 0, None), ("odd split", (1, 11), 0, None),
                                     ("one by one", (1,) * 12, 0, None), ("diagnostics", (12,), 5, None),
                                     ("every step", (12,), 1, None), ("one cell", (12,), 0, (1, 128)), ("one cell, diagnostics", (12,), 1, (1, 128))):
        lat = lbm.Lattice(D - 2, dims, 0.6, eq, bulk, lbm.F64)
        if shape:
            lat.set_launch_shape(*shape)
        lat.set_option(lbm.OPT_DIAG_EVERY, diag)
        lat.init_fields(rho, u)
        for n in calls:
            lat.step(n)
        got[name] = lat.get_populations("storage")
        lat.close()
    for name, f in got.items():
        assert np.array_equal(f, got["several"]), name


def test_checkpoint_at_any_step():
    """The documented checkpoint (stored values and step count), taken after any number of steps."""
    from paper_2303_08163_gb300 import lbm
    dims = (64, 64, 1)
    rho, u = inputs.taylor_green_2d(64, u0=0.05)
    whole = lbm.Lattice(lbm.D2Q9, dims, 0.8, lbm.ENTROPIC, 1, lbm.F64)
    whole.init_fields(rho, u)
    whole.step(100)
    for first in (1, 2, 50, 99):
        a = lbm.Lattice(lbm.D2Q9, dims, 0.8, lbm.ENTROPIC, 1, lbm.F64)
        a.init_fields(rho, u)
        a.step(first)
        b = lbm.Lattice(lbm.D2Q9, dims, 0.8, lbm.ENTROPIC, 1, lbm.F64)
        b.set_step_count(a.step_count)
        b.set_populations(a.get_populations("storage"), "storage")
        b.step(100 - first)
        assert np.array_equal(b.get_populations("storage"), whole.get_populations("storage")), first
        a.close()
        b.close()
    whole.close()


@pytest.mark.parametrize("eq,bulk", EQS)
@pytest.mark.parametrize("D,dims", [(2, [(128, 1, 1)] * 28), (2, [(90, 80, 1), (3, 2, 1), (16, 16, 1)]), (3, [(16, 9, 1), (4, 5, 6)]),
                                    (3, [(20, 22, 24), (5, 4, 3)])])
def test_batch(D, dims, eq, bulk):
    from paper_2303_08163_gb300 import lbm
    dims = np.array(dims, dtype=np.int32)
    n = len(dims)
    tau = 0.5 + np.random.default_rng(n).uniform(0.05, 0.5, n)
    fields = [inputs.random_state(D, tuple(int(v) for v in d), seed=20 + i, u_max=0.1) for i, d in enumerate(dims)]
    rho = np.concatenate([f[0] for f in fields])
    u = np.concatenate([f[1].reshape(-1) for f in fields])
    got = []
    for whole, every, calls in ((False, 0, (11,)), (False, 2, (6, 5)), (True, 0, (11,)), (True, 3, (1, 10))):
        b = lbm.Batch(lbm.D2Q9 if D == 2 else lbm.D3Q27, dims, tau, eq, bulk)
        if whole:
            b.set_launch_shape(64, min(n, 3))
        b.init_fields(rho, u)
        if every:
            b.set_probe(np.array([(1, 0, 0)] * n, dtype=np.int32), every)
        for steps in calls:
            b.step(steps)
        got.append(b.get_populations())
        b.close()
    for f in got[1:]:
        assert np.array_equal(f, got[0])

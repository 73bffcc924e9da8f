"""Several steps in one launch of the TMA row kernel (job tickets, done counters, several steps
in flight) against one launch per step of the one-cell kernel on the same stored values."""
import numpy as np
import pytest

from paper_2303_08163_gb300 import inputs

pytestmark = pytest.mark.gpu

# (D, dims, precision, shape or None): fewer positions than neighbours, one position, several
# jobs a position, segments, padded rows, more jobs than blocks, short last row groups
CASES = [
    (2, (64, 64, 1), 0, None), (2, (64, 1, 1), 0, None), (2, (64, 2, 1), 1, None), (2, (48, 3, 1), 2, None),
    (2, (256, 700, 1), 1, (2, 128, 2, 1, 64, 1024)), (2, (509, 381, 1), 1, None), (2, (40, 37, 1), 2, (2, 64, 3, 4, 40, 1024)),
    (3, (32, 32, 32), 2, None), (3, (16, 9, 1), 1, None), (3, (16, 5, 2), 2, None), (3, (16, 40, 3), 0, None),
    # the largest lattice of the grid-barrier kernel on 152 SMs, and the next one
    (2, (320, 380, 1), 1, None), (2, (320, 381, 1), 1, None), (3, (64, 50, 38), 2, None), (3, (61, 53, 37), 1, None),
    (3, (64, 30, 31), 1, None), (3, (67, 20, 11), 2, None), (3, (96, 64, 20), 2, (2, 128, 2, 1, 48, 1024)),
]


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("D,dims,prec", [(3, (256, 40, 24), 2), (3, (128, 40, 24), 1), (2, (512, 500, 1), 2),
                                         (2, (512, 500, 1), 1)])
def test_pairs_store_the_bits_of_single_cells(D, dims, prec, eq, bulk):
    """The packed two-cell FP32 collision against the one-cell one, both parities."""
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=80 + eq, u_max=0.15)
    lats = [lbm.Lattice(D - 2, dims, 0.6, eq, bulk, prec) for _ in range(2)]
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 256)
    for lat in lats:
        lat.init_fields(rho, u)
    for _ in range(2):
        for lat in lats:
            lat.step(1)
        assert np.array_equal(*(lat.get_populations("storage") for lat in lats))
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("D,dims,prec,shape", CASES)
def test_many_steps_match_single_steps(D, dims, prec, shape):
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=70 + dims[1], rho_range=(0.9, 1.1), u_max=0.05)
    lats = [lbm.Lattice(D - 2, dims, 0.7, 0, 1, prec) for _ in range(2)]
    if shape:
        lats[0].set_launch_shape(*shape)
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 128)
    for lat in lats:
        lat.init_fields(rho, u)
    assert lats[0].launch_info()["kernel"] == lbm.KERNEL_TMA
    # both parities at the start of a launch, one step, many, repeated launches
    for n in (2, 3, 1, 40, 17):
        for lat in lats:
            lat.step(n)
        a, b = (lat.get_populations("storage") for lat in lats)
        if prec == 0:
            assert np.max(np.abs(a - b)) <= 1e-14
        else:
            assert np.array_equal(a, b)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("D,dims,prec", [(3, (256, 64, 130), 2), (3, (130, 128, 70), 1), (2, (1024, 3000, 1), 1),
                                         (2, (4096, 1500, 1), 2)])
def test_states_larger_than_l2(D, dims, prec):
    """Swept several steps at a time; a diagnostics period that splits the launches."""
    import torch
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state_torch(D, dims, seed=5, u_max=0.05)
    lats = [lbm.Lattice(D - 2, dims, 0.6, 0, 0, prec) for _ in range(2)]
    lats[1].set_launch_shape(lbm.KERNEL_GENERIC, 128)
    for lat in lats:
        lat.init_fields(rho, u, dtype=np.float32)
    st = {1: torch.float32, 2: torch.float16}[prec]
    for n in (9, 6, 2):
        for lat in lats:
            lat.step(n)
        a, b = (lat.get_populations("storage", out=torch.empty((lat.Q, lat.ncell), dtype=st, device="cuda")) for lat in lats)
        assert torch.equal(a, b)
    for lat in lats:
        lat.set_option(lbm.OPT_DIAG_EVERY, 5)
        lat.step(13)
    a, b = (lat.get_populations("storage", out=torch.empty((lat.Q, lat.ncell), dtype=st, device="cuda")) for lat in lats)
    assert torch.equal(a, b)
    assert [d["step"] for d in lats[0].diag_history()] == [20, 25]
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("D,dims,prec", [(2, (96, 70, 1), 0), (3, (40, 24, 20), 2), (3, (96, 80, 70), 2)])
def test_steps_inside_a_stream_capture(D, dims, prec):
    """lbm_step recorded in a caller's graph and replayed."""
    import torch
    from paper_2303_08163_gb300 import lbm
    rho, u = inputs.random_state(D, dims, seed=31, u_max=0.05)
    s = torch.cuda.Stream()
    lats = [lbm.Lattice(D - 2, dims, 0.7, 0, 0, prec, stream=s) for _ in range(2)]
    for lat in lats:
        lat.init_fields(rho, u)
        lat.step(6)
        lat.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        lats[0].step(6)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    lats[1].step(18)
    assert np.array_equal(*(lat.get_populations("storage") for lat in lats))
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("dims", [(128, 128, 24), (32, 32, 32)])
def test_lattices_on_two_streams(dims):
    """Two lattices stepping at once on their own streams: launches that wait for their own
    blocks' counters only."""
    import torch
    from paper_2303_08163_gb300 import lbm
    streams = [torch.cuda.Stream() for _ in range(2)]
    rho, u = inputs.random_state(3, dims, seed=9, u_max=0.05)
    lats = [lbm.Lattice(1, dims, 0.6, 0, 0, 2, stream=s) for s in streams]
    for lat in lats:
        lat.init_fields(rho, u)
    for _ in range(20):
        for lat in lats:
            lat.step(25)
    got = [lat.get_populations("storage") for lat in lats]
    assert np.array_equal(got[0], got[1])
    ref = lbm.Lattice(1, dims, 0.6, 0, 0, 2)
    ref.set_launch_shape(lbm.KERNEL_GENERIC, 256)
    ref.init_fields(rho, u)
    ref.step(500)
    assert np.array_equal(got[0], ref.get_populations("storage"))
    for lat in lats + [ref]:
        lat.close()

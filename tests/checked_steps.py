"""Cases of tests/test_gpu_checked_steps.py, run by it against the bounds-checked library in a child
process: the kernels of several steps (TMA row kernel, small lattices, three lanes a cell) and of batches
(whole instances, teams, clusters), and the transfers of padded rows."""
import sys

import numpy as np

from paper_2303_08163_gb300 import inputs

# (D, dims, precision, launch shape or None)
LATTICES = [
    (2, (64, 3, 1), 1, (2, 64, 2, 1, 64, 1024)), (2, (200, 33, 1), 2, (2, 96, 3, 1, 72, 1024)), (2, (131, 9, 1), 2, (2, 128, 2, 2, 131, 1024)),
    (2, (40, 18, 1), 0, (2, 128, 2, 4, 40, 2048)), (3, (16, 9, 1), 1, (2, 64, 2, 2, 16, 1024)), (3, (48, 20, 9), 2, (2, 128, 2, 3, 48, 1024)),
    (3, (67, 6, 5), 2, (2, 128, 2, 2, 67, 1024)), (3, (96, 6, 4), 2, (2, 128, 2, 1, 48, 1024)), (3, (33, 5, 4), 1, (2, 128, 2, 3, 33, 1024)),
    (2, (1, 1, 1), 0, None), (2, (3, 1, 1), 1, None), (2, (41, 37, 1), 0, None), (2, (131, 97, 1), 2, None), (2, (160, 150, 1), 0, None),
    (2, (509, 381, 1), 1, None), (3, (1, 2, 3), 2, None), (3, (7, 11, 13), 0, None), (3, (31, 40, 31), 2, None), (3, (29, 32, 76), 1, None),
    (3, (30, 31, 33), 0, None), (3, (48, 48, 50), 0, None), (3, (301, 40, 30), 2, None), (2, (2047, 300, 1), 1, None), (2, (1024, 2100, 1), 1, None),
]
BATCHES = [(2, [(128, 1, 1)] * 5 + [(9, 11, 1), (1, 1, 1)]), (2, [(90, 80, 1), (3, 2, 1), (16, 16, 1)]), (3, [(16, 9, 1), (1, 1, 1), (4, 5, 6)]),
           (3, [(20, 22, 24), (5, 4, 3)]), (2, [(12 + k % 30, 9 + k % 21, 1) for k in range(160)])]


def run(lbm, out_path):
    res = {}
    for n, (D, dims, prec, shape) in enumerate(LATTICES):
        rho, u = inputs.random_state(D, dims, seed=700 + n, u_max=0.1)
        lat = lbm.Lattice(D - 2, dims, 0.6, n % 3, n % 2, prec)
        if shape:
            lat.set_launch_shape(*shape)
        lat.init_fields(rho, u)
        for t, k in enumerate((2, 3, 1, 8)):
            lat.step(k)
            lat.sync()
            res[f"lat{n}_{t}"] = lat.get_populations("storage").view(np.uint8)
        lat.set_populations(lat.get_populations(np.float32), np.float32)
        lat.set_option(lbm.OPT_DIAG_EVERY, 2)
        lat.step(3)
        lat.sync()
        res[f"lat{n}_io"] = lat.get_populations("storage").view(np.uint8)
        lat.close()
    for n, (D, dims) in enumerate(BATCHES):
        dims = np.array(dims, dtype=np.int32)
        fields = [inputs.random_state(D, tuple(int(v) for v in d), seed=60 + i, u_max=0.1) for i, d in enumerate(dims)]
        for whole in (0, 1):
            b = lbm.Batch(D - 2, dims, np.linspace(0.6, 0.9, len(dims)), n % 3, n % 2)
            if whole:
                b.set_launch_shape(64, min(len(dims), 3))
            b.init_fields(np.concatenate([f[0] for f in fields]), np.concatenate([f[1].reshape(-1) for f in fields]))
            b.set_probe(np.array([(1, 0, 0)] * len(dims), dtype=np.int32), 2)
            for k in (3, 1, 4):
                b.step(k)
            b.sync()
            assert not b.status().any(), (n, whole, b.status())
            res[f"batch{n}_{whole}"] = b.get_populations().view(np.uint8)
            b.close()
    np.savez(out_path, **res)


if __name__ == "__main__":
    from paper_2303_08163_gb300 import lbm as _lbm
    _lbm.load()
    run(_lbm, sys.argv[1])

"""The FP64 collisions where their shorter forms could leave the formulas: negative and zero density,
densities near the ends of FP64's range, and the reciprocal and square root by themselves."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import core

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
W1 = np.array([1 / 6, 2 / 3, 1 / 6])


def weights(D):
    w = np.multiply.outer(W1, W1) if D == 2 else np.multiply.outer(W1, np.multiply.outer(W1, W1))
    return w.reshape(-1, 1)


def velocities(D):
    g = np.arange(-1, 2)
    c = np.array(np.meshgrid(*[g] * D, indexing="ij")).reshape(D, -1)[::-1]  # x fastest
    return c.astype(np.float64)


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 1), (2, 1)])
@pytest.mark.parametrize("D,dims", [(2, (16, 9, 1)), (2, (131, 97, 1)), (3, (8, 5, 7)), (3, (24, 26, 28))])
def test_negative_density(D, dims, eq, bulk):
    """States that overshoot: cells of density -0.05, some of them without momentum."""
    from paper_2303_08163_gb300 import lbm
    n, c, w = int(np.prod(dims)), velocities(D), weights(D)
    rng = np.random.default_rng(n)
    rho = np.where(rng.random(n) < 0.3, -0.05, 1.0)
    u = rng.uniform(-0.4, 0.4, (D, n)) * (rng.random(n) < 0.7)
    f = w * rho * (1 + 3 * (c.T @ u))
    ref = core.step(D, dims, eq, bulk, 0.8, 1, f)
    # |f| < 1: some 40 roundings of values below 1, those of rho = -0.05 twenty times as large in u
    tol = 20 * 40 * 2.0 ** -54
    for shape in (None, (lbm.KERNEL_GENERIC, 64)):
        lat = lbm.Lattice(D - 2, dims, 0.8, eq, bulk, lbm.F64)
        if shape:
            lat.set_launch_shape(*shape)
        lat.set_populations(f)
        lat.step(1)
        assert np.max(np.abs(lat.get_populations() - ref)) <= tol
        lat.close()


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 1), (2, 1)])
@pytest.mark.parametrize("D,dims", [(2, (16, 9, 1)), (2, (131, 97, 1)), (3, (8, 5, 7)), (3, (24, 26, 28))])
@pytest.mark.parametrize("v", [(0.3, -0.2, 0.1), (0.0, 0.0, 0.0)])
def test_uniform_negative_density_stays(D, dims, eq, bulk, v):
    """A uniform flow of negative density is at its equilibrium: the kernels of several steps and of
    batches (clusters, teams) keep it there."""
    from paper_2303_08163_gb300 import lbm
    n, steps = int(np.prod(dims)), 9
    rho, u = np.full(n, -0.05), np.repeat(np.array(v[:D]), n).reshape(D, n)
    want = core.init(D, dims, eq, rho, u)
    tol = steps * 20 * 40 * 2.0 ** -54  # as above, a step
    lat = lbm.Lattice(D - 2, dims, 0.8, eq, bulk, lbm.F64)
    lat.set_populations(want)
    lat.step(steps)
    assert np.max(np.abs(lat.get_populations() - want)) <= tol
    lat.close()
    for extra in ([], [(3, 2, 1)]):
        b = lbm.Batch(D - 2, np.array([dims] + extra, dtype=np.int32), np.full(1 + len(extra), 0.8), eq, bulk)
        m = sum(a * c for a, c, _ in extra)
        b.init_fields(np.full(n + m, -0.05), np.concatenate([u.ravel(), np.repeat(np.array(v[:D]), m)]))
        b.step(steps)
        assert np.max(np.abs(b.get_populations()[:want.size].reshape(want.shape) - want)) <= tol
        b.close()


@pytest.mark.parametrize("eq,bulk", [(0, 0), (0, 1), (1, 1), (2, 0)])
@pytest.mark.parametrize("D,dims", [(2, (20, 9, 1)), (2, (100, 97, 1)), (3, (6, 5, 7)), (3, (24, 25, 22))])
def test_densities_of_any_size(D, dims, eq, bulk):
    """The scheme is homogeneous: a power of two in the density changes the exponents and nothing else."""
    from paper_2303_08163_gb300 import inputs, lbm
    rho, u = inputs.random_state(D, dims, seed=4, rho_range=(0.9, 1.1), u_max=0.15)

    def run(scale, steps):
        lat = lbm.Lattice(D - 2, dims, 0.6, eq, bulk, lbm.F64, rho0=scale)
        lat.init_fields(rho * scale, u)
        for n in steps:
            lat.step(n)
        f = lat.get_populations()
        lat.close()
        return f / scale

    for steps in ((1,), (3,)):
        want = run(1.0, steps)
        assert np.isfinite(want).all()
        for k in (-960, -500, -345, -260, 260, 345, 500, 960):
            assert np.array_equal(run(2.0 ** k, steps), want), k


@pytest.mark.parametrize("dims", [[(12, 9, 1), (40, 3, 1)], [(90, 80, 1), (3, 2, 1)]])
def test_batches_of_any_density(dims):
    from paper_2303_08163_gb300 import inputs, lbm
    dims = np.array(dims, dtype=np.int32)
    fields = [inputs.random_state(2, tuple(int(v) for v in d), seed=5, u_max=0.1) for d in dims]
    rho = np.concatenate([f[0] for f in fields])
    u = np.concatenate([f[1].reshape(-1) for f in fields])
    got = []
    for scale in (1.0, 2.0 ** -400, 2.0 ** 400):
        b = lbm.Batch(lbm.D2Q9, dims, np.array([0.6, 0.8]), lbm.ENTROPIC, 1, rho0=scale)
        b.init_fields(rho * scale, u)
        b.step(5)
        got.append(b.get_populations() / scale)
        b.close()
    assert np.isfinite(got[0]).all()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


KERNEL = r"""
#include "lbm_device.cuh"
__global__ void k(const double *x, double *r, double *s, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = lbmd::rcp_any(x[i]);
    s[i] = lbmd::sqrt_ulp(x[i]);
}
extern "C" int run(const double *x, double *r, double *s, int n) {
    double *d = nullptr;
    if (cudaMalloc(&d, 3 * sizeof(double) * n) != cudaSuccess) return 1;
    cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
    cudaMemcpy(r, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(s, d + 2 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)cudaGetLastError();
}
"""


def test_reciprocal_and_square_root(tmp_path):
    """Within an ulp of the correctly rounded values wherever x and 1/x are normal numbers (the iteration
    leaves 2^-60 and half an ulp of rounding, the square root another half); 1/0 and 1/NaN are not finite
    or, like 1/infinity, below the normal numbers."""
    from paper_2303_08163_gb300 import build
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    (tmp_path / "k.cu").write_text(KERNEL)
    r = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                        str(tmp_path / "k.cu"), "-o", str(tmp_path / "k.so")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    fn = ctypes.CDLL(str(tmp_path / "k.so")).run
    rng = np.random.default_rng(6)
    e = rng.integers(-1022, 1024, 400000)
    x = np.ldexp(rng.uniform(1, 2, len(e)), e)
    edge = np.ldexp(np.array([1.0, 1 + 2.0 ** -52, 1.5, 2 - 2.0 ** -52]), np.arange(-1022, 1024)[:, None]).ravel()
    special = np.array([0.0, np.inf, np.nan, 5e-324, 2.2e-308, 1e-310, np.finfo(float).max, np.finfo(float).tiny])
    x = np.concatenate([x, -x[:1000], edge, special, -special])
    rc, sq = np.zeros_like(x), np.zeros_like(x)
    dbl = ctypes.POINTER(ctypes.c_double)
    assert fn(x.ctypes.data_as(dbl), rc.ctypes.data_as(dbl), sq.ctypes.data_as(dbl), ctypes.c_int(len(x))) == 0
    with np.errstate(all="ignore"):
        want = 1.0 / x
        tiny = np.finfo(float).tiny
        normal = np.isfinite(x) & (np.abs(x) >= tiny)
        both = normal & (np.abs(want) >= tiny)
        assert np.all(np.abs(rc - want)[both] <= np.spacing(np.abs(want[both])))
        assert np.all(np.isnan(rc[np.abs(x) < tiny])) and np.all(np.abs(rc[np.isinf(x)]) < tiny)
        pos = normal & (x > 0)
        root = np.sqrt(x[pos])
        assert np.all(np.abs(sq[pos] - root) <= np.spacing(root))


@pytest.mark.parametrize("eq", [0, 1, 2])
def test_huge_relaxation_time(eq):
    """No relaxation at all, with the corrected rate too: populations only stream."""
    from paper_2303_08163_gb300 import inputs, lbm
    dims = (20, 9, 1)
    rho, u = inputs.random_state(2, dims, seed=2, u_max=0.1)
    for tau in (1e200, 1.7e308):
        for bulk in (0, 1):
            lat = lbm.Lattice(lbm.D2Q9, dims, tau, eq, bulk, lbm.F64)
            lat.init_fields(rho, u)
            f0 = lat.get_populations("storage")
            for n, back in ((1, 1), (2, 3)):
                lat.step(n)
                f = lat.get_populations("storage")
                for i, c in enumerate(velocities(2).T.astype(int)):
                    want = np.roll(f0[i].reshape(9, 20), (c[1] * back, c[0] * back), axis=(0, 1)).ravel()
                    assert np.array_equal(f[i], want)
            lat.close()

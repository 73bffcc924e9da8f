"""The stability search with and without its look-ahead takes the decisions of plain bisection, and does
not take longer than solving every trial's sweep."""
import math
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def bisect(lbm, eq, nu, th, nk, u_hi, iterations, tol):
    n, k = len(nu), math.pi * np.arange(nk) / (nk - 1)
    kx, ky = (v.ravel() for v in np.meshgrid(k, k))

    def stable(u):
        p = np.empty((n, nk * nk, 6))
        p[:, :, 0], p[:, :, 1], p[:, :, 4], p[:, :, 5] = (0.5 + 3 * nu)[:, None], 1.0, kx, ky
        p[:, :, 2], p[:, :, 3] = (u * np.cos(th))[:, None], (u * np.sin(th))[:, None]
        return np.abs(lbm.vn_eigenvalues(eq, 0, p.reshape(-1, 6))).reshape(n, -1).max(1) <= 1 + tol

    lo, hi, top = np.zeros(n), np.full(n, u_hi), stable(np.full(n, u_hi))
    for _ in range(iterations):
        mid = 0.5 * (lo + hi)
        s = stable(mid)
        lo, hi = np.where(s, mid, lo), np.where(s, hi, mid)
    return np.where(top, u_hi, lo)


# sweeps below, at and above eight look-aheads; few pairs, which have the GPU to themselves
@pytest.mark.parametrize("eq", [0, 1, 2])
@pytest.mark.parametrize("pairs,nk", [(700, 3), (40, 15), (40, 16), (40, 17), (20, 6), (101, 7)])
def test_decisions(eq, pairs, nk):
    from paper_2303_08163_gb300 import lbm
    rng = np.random.default_rng(pairs + nk)
    nu, th = 10.0 ** rng.uniform(-3, 0, pairs), rng.uniform(0.05, 1.5, pairs)
    got = lbm.vn_stability_limit(eq, nu, th, nk=nk, u_hi=0.9, iterations=13, tol=1e-7)
    assert np.array_equal(got, bisect(lbm, eq, nu, th, nk, 0.9, 13, 1e-7))


def test_small_sweeps_take_no_longer_than_all_their_trials():
    from paper_2303_08163_gb300 import lbm
    rng = np.random.default_rng(5)
    pairs, nk, iterations = 2000, 3, 14
    nu, th = 10.0 ** rng.uniform(-3, 0, pairs), rng.uniform(0.05, 1.5, pairs)
    params = np.ones((pairs * nk * nk, 6)) * (0.6, 1.0, 0.2, 0.1, 1.0, 0.7)

    def least(f):
        f()
        best = math.inf
        for _ in range(4):
            t = time.perf_counter()
            f()
            best = min(best, time.perf_counter() - t)
        return best

    trial = least(lambda: lbm.vn_eigenvalues(1, 0, params))
    search = least(lambda: lbm.vn_stability_limit(1, nu, th, nk=nk, u_hi=0.9, iterations=iterations, tol=1e-7))
    assert search <= 1.25 * (iterations + 1) * trial, (search, trial)

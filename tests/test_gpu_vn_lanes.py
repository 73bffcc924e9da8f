"""von Neumann kernels over their launch forms: the number of lanes a matrix gets depends on the
size of the call and must not change a result; the look-ahead of the stability search must not
change a decision."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def points(n, seed):
    rng = np.random.default_rng(seed)
    return np.stack([0.5 + 10 ** rng.uniform(-4, 0.3, n), rng.uniform(0.9, 1.1, n), rng.uniform(-0.3, 0.3, n),
                     rng.uniform(-0.3, 0.3, n), rng.uniform(0, math.pi, n), rng.uniform(0, math.pi, n)], axis=1)


@pytest.mark.parametrize("eq,bulk", [(0, 0), (1, 1), (2, 0)])
def test_spectra_do_not_depend_on_the_call_size(eq, bulk):
    from paper_2303_08163_gb300 import lbm
    p = points(20001, 3 + eq)                                   # one lane a matrix
    whole = lbm.vn_eigenvalues(eq, bulk, p)
    for n in (1, 7, 8, 33, 4864, 4865, 19456):                  # four lanes, two lanes
        assert np.array_equal(lbm.vn_eigenvalues(eq, bulk, p[:n]), whole[:n]), n


@pytest.mark.parametrize("eq", [0, 1, 2])
@pytest.mark.parametrize("pairs,nk,iterations", [(3, 5, 9), (40, 24, 12), (2, 1, 3)])
def test_search_takes_the_decisions_of_plain_bisection(eq, pairs, nk, iterations):
    from paper_2303_08163_gb300 import lbm
    rng = np.random.default_rng(17 + pairs)
    nu, th = 10.0 ** rng.uniform(-3, 0, pairs), rng.uniform(0.05, 1.5, pairs)
    u_hi, tol = 0.9, 1e-7
    got = lbm.vn_stability_limit(eq, nu, th, nk=nk, u_hi=u_hi, iterations=iterations, tol=tol)
    k = math.pi * np.arange(nk) / (nk - 1) if nk > 1 else np.zeros(1)
    kx, ky = (v.ravel() for v in np.meshgrid(k, k))

    def stable(u):
        r = [np.abs(lbm.vn_eigenvalues(eq, 0, np.stack([np.full(nk * nk, 0.5 + 3 * nu[i]), np.ones(nk * nk),
                                                        np.full(nk * nk, u[i] * np.cos(th[i])),
                                                        np.full(nk * nk, u[i] * np.sin(th[i])), kx, ky], 1))).max()
             for i in range(pairs)]
        return np.array(r) <= 1 + tol

    lo, hi = np.zeros(pairs), np.full(pairs, u_hi)
    top = stable(hi)
    for _ in range(iterations):
        mid = 0.5 * (lo + hi)
        s = stable(mid)
        lo, hi = np.where(s, mid, lo), np.where(s, hi, mid)
    assert np.array_equal(got, np.where(top, u_hi, lo))

"""Evaluations do not depend on the unit of length: coordinates times 2^k with eps and psi times 2^2k give the
same gradient, also where squared distances or 1/eps leave FP32's range.

The mixed passes' operands scale by powers of two exactly, so their results keep their bits.  FP64: the
exponents' rounding in the general passes (2^-53 of terms up to 1,500 here, in each pass) and sums.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(d, nq, n, seed):
    rng = np.random.default_rng(seed)
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    return rng.uniform(0, 1, (nq, d)), m / m.sum(), rng.uniform(0, 1, (n, d)), nu / nu.sum(), rng


def _eval(x, m, y, nu, psi, eps, k, prec, kind=None):
    import paper_2507_23602_gb300 as rs
    s = 2.0 ** k
    P = rs.Problem(x * s, m, y * s, nu)
    try:
        if kind is not None:
            P.set_pair_kernel(kind)
        J, g, _ = P.eval(psi * s * s, eps * s * s, 0.0, prec)
        return J / (s * s), g
    finally:
        P.close()


@pytest.mark.parametrize("k", [-80, -70, -40, -20, 20, 40, 64, 70, 200])
def test_fp64(k):
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, rng = _problem(3, 3000, 700, 1)
    psi, eps = 1e-3 * rng.standard_normal(700), 1e-3
    J, g = _eval(x, m, y, nu, psi, eps, 0, rs.FP64)
    Jk, gk = _eval(x, m, y, nu, psi, eps, k, rs.FP64)
    assert np.all(np.abs(gk - g) <= 1e-11 * (g + 2 * nu)) and abs(J - Jk) <= 1e-12 * abs(J)


# points by cells, whose warps keep finite boxes where the distances to most targets overflow
@pytest.mark.parametrize("k", [-80, -34, 49, 51, 66, 68])
def test_fp64_points_by_cells(k):
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, rng = _problem(3, 24576, 500, 4)
    x = x[np.lexsort(np.floor(8 * x).T)]
    psi, eps = 1e-3 * rng.standard_normal(500), 1e-3
    J, g = _eval(x, m, y, nu, psi, eps, 0, rs.FP64)
    Jk, gk = _eval(x, m, y, nu, psi, eps, k, rs.FP64)
    assert np.all(np.abs(gk - g) <= 1e-11 * (g + 2 * nu)) and abs(J - Jk) <= 1e-12 * abs(J)


@pytest.mark.parametrize("k", [-60, -40, -20, 20, 40, 50])
def test_compensated(k):
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, rng = _problem(3, 3000, 1500, 2)
    psi, eps = 1e-3 * rng.standard_normal(1500), 1e-3
    J, g = _eval(x, m, y, nu, psi, eps, 0, rs.COMPENSATED)
    Jk, gk = _eval(x, m, y, nu, psi, eps, k, rs.COMPENSATED)
    assert np.all(np.abs(gk - g) <= 2 * 6.0e-7 * (g + nu) + 1e-14 * nu)
    assert abs(J - Jk) <= 2 * 3e-7 * eps + 1e-13 * abs(J)


@pytest.mark.parametrize("k", [-62, -55, -20, 20, 45, 60])
def test_mixed_that_leaves_out_pairs(k):
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, rng = _problem(3, 98304, 16384, 3)
    psi, eps = 5e-4 * rng.standard_normal(16384), 1e-3
    J, g = _eval(x, m, y, nu, psi, eps, 0, rs.MIXED, rs.PAIRS_FP32)
    Jk, gk = _eval(x, m, y, nu, psi, eps, k, rs.MIXED)
    # FP64 sums in another order (test_mskip_gpu.py)
    assert np.all(np.abs(gk - g) <= (98304 / 512 + 2) * 2.0 ** -52 * (g + 2 * nu))
    assert abs(Jk - J) <= 2.0 ** -50 * (1 + abs(J))

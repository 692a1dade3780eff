"""Compensated dense evaluations returned to a caller (rsot_cx.cu) against the FP64 evaluation.

Tolerance: the evaluation's certified bound, 6.0e-7 of a target's transported mass per entry and
6.5e-7 of the mass in the L1 norm (J: 3e-7 eps sum m).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(d, nq, n, seed, zero_mass=False, scale=1.0):
    rng = np.random.default_rng(seed)
    x = scale * rng.uniform(0, 1, (nq, d))
    m = rng.uniform(0.2, 1.8, nq)
    if zero_mass:
        m[1::4] = 0.0
    y = scale * rng.uniform(0, 1, (n, d))
    nu = rng.uniform(0.5, 1.5, n) * 10.0 ** rng.uniform(-3, 0, n)
    return x, m / m.sum(), y, nu / nu.sum(), rng


def _check(d, nq, n, eps, spread, seed, form="grad_cx", psi=None, **kw):
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, rng = _problem(d, nq, n, seed, **kw)
    if psi is None:
        psi = spread * rng.standard_normal(n)
    P = rs.Problem(x, m, y, nu)
    try:
        J64, g64, _ = P.eval(psi, eps, 0.0, rs.FP64)
        L64 = P.point_log_partition()
        P.kernel_timing(True)
        J, g, pairs = P.eval(psi, eps, 0.0, rs.COMPENSATED)
        names = set(P.kernel_times())
        L = P.point_log_partition()
    finally:
        P.close()
    assert form in names and pairs == nq * n
    a = g64 + nu
    assert np.all(np.abs(g - g64) <= 6.0e-7 * a + 1e-14 * nu)
    assert np.abs(g - g64).sum() <= rs.COMPENSATED_GRAD_REL
    assert abs(J - J64) <= 3e-7 * eps + 1e-13 * abs(J64)
    assert np.max(np.abs(L - L64)) <= 3e-7 + 1e-13 * np.max(np.abs(L64))


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("nq,n", [(1, 1000), (255, 1001), (257, 1153), (1025, 1023), (2049, 2500)])
def test_sizes(d, nq, n):
    _check(d, nq, n, 1e-2, 0.005, seed=nq + n)


@pytest.mark.parametrize("eps,spread", [(0.5, 0.3), (1e-3, 0.005), (1e-3, 0.4), (1e-4, 0.02)])
def test_ranges_of_the_exponent(eps, spread):
    _check(3, 3000, 1500, eps, spread, seed=5)


def test_points_without_mass_and_large_coordinates():
    _check(2, 1600, 1201, 5e-3, 0.01, seed=6, zero_mass=True)
    _check(3, 900, 1100, 1e4, 500.0, seed=7, scale=1.0e3)


def test_constants_beyond_the_exact_sums_take_the_general_passes():
    psi = 0.01 * np.random.default_rng(8).standard_normal(1100)
    psi[17] = 40.0
    _check(2, 700, 1100, 1e-2, 0.0, seed=9, form="grad_df", psi=psi)


def test_solves_keep_the_general_passes():
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, _ = _problem(2, 1500, 1024, 10)
    P = rs.Problem(x, m, y, nu)
    try:
        P.kernel_timing(True)
        P.solve(eps=2e-2, tol_l1=1e-4, precision=rs.COMPENSATED)
        names = set(P.kernel_times())
    finally:
        P.close()
    assert "grad_df" in names and "grad_cx" not in names


# from 1e9 pairs on the points' maxima leave out targets and the points are taken in cell order by pairs:
# an odd number of points in no order, one chunk of targets and many, clusters apart
@pytest.mark.parametrize("d,nq,n,eps", [(3, 100001, 10007, 1e-3), (2, 400003, 2503, 1e-3), (3, 5121, 200001, 2e-3)])
def test_large(d, nq, n, eps):
    _check(d, nq, n, eps, 2 * eps, seed=nq)

"""Dense FP64 evaluation with fixed-point exponents (rsot_fx64.cu) against extended precision.

Tolerance: the integer exponent is within 6 units of 2^-F <= 2^-46 (2^-52 except where the
exponents are large) and the column sums of at most 4,096 FP64 terms round by at most
4,096 * 2^-53 = 4.6e-13, in each of the two passes: an entry errs by less than 1e-12 of the
larger of its transported mass and nu_j.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _exact(x, m, y, nu, psi, eps):
    x, m, y, nu, psi = (np.asarray(v).astype(LD) for v in (x, m, y, nu, psi))
    eps = LD(eps)
    a = np.zeros(len(nu), LD)
    J = -(psi * nu).sum()
    L = np.empty(len(x), LD)
    for q in range(0, len(x), 64):
        c = ((x[q:q + 64, None, :] - y[None]) ** 2).sum(-1) / 2
        s = (psi[None] - c) / eps + np.log(nu)[None]
        top = s.max(1)
        p = np.exp(s - top[:, None])
        S = p.sum(1)
        L[q:q + 64] = top + np.log(S)
        J += (m[q:q + 64] * eps * L[q:q + 64]).sum()
        a += ((m[q:q + 64] / S)[:, None] * p).sum(0)
    return J, a, L


def _names(P):
    return set(P.kernel_times())


def _check(d, nq, n, eps, spread, seed, fixed_point=True, zero_mass=False, scale=1.0):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(seed)
    x = scale * rng.uniform(0, 1, (nq, d))
    m = rng.uniform(0.2, 1.8, nq)
    if zero_mass:
        m[::3] = 0.0
        m[1] = 1.0
    m /= m.sum()
    y = scale * rng.uniform(0, 1, (n, d))
    nu = rng.uniform(0.5, 1.5, n) * 10.0 ** rng.uniform(-4, 0, n)
    nu /= nu.sum()
    psi = spread * rng.standard_normal(n)
    P = rs.Problem(x, m, y, nu)
    try:
        P.kernel_timing(True)
        J, g, pairs = P.eval(psi, eps, 0.0, rs.FP64)
        names = _names(P)
        L = P.point_log_partition()
    finally:
        P.close()
    assert ("fx_grad" in names) and (("grad_fp64" in names) != fixed_point)
    assert pairs == nq * n
    Je, a, Le = _exact(x, m, y, nu, psi, eps)
    tol = 1e-12 if fixed_point else 1e-10
    assert abs(LD(J) - Je) <= tol * (abs(Je) + LD(eps) * np.abs(m * Le).sum())
    err = np.abs(g.astype(LD) - (a - nu.astype(LD)))
    assert np.all(err <= tol * np.maximum(a, nu)), float((err / np.maximum(a, nu)).max())
    assert np.all(np.abs(L.astype(LD) - Le) <= tol * np.maximum(1, np.abs(Le)))


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("nq,n", [(1, 1), (2, 129), (127, 2), (129, 128), (1025, 127), (515, 1025)])
def test_sizes(d, nq, n):
    _check(d, nq, n, 1e-2, 0.005, seed=nq + n)


@pytest.mark.parametrize("eps,spread", [(0.5, 0.3), (1e-3, 0.005), (1e-3, 0.4), (1e-4, 0.02)])
def test_ranges_of_the_exponent(eps, spread):
    _check(3, 700, 300, eps, spread, seed=5)


def test_points_without_mass():
    _check(2, 600, 257, 5e-3, 0.01, seed=6, zero_mass=True)


def test_large_coordinates():
    _check(3, 400, 200, 1e4, 500.0, seed=7, scale=1.0e3)


def test_exponents_beyond_the_fixed_point_range_take_the_fp64_passes():
    _check(2, 300, 200, 1e-6, 40.0, seed=8, fixed_point=False)


def test_non_finite_potential_is_refused():
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(9)
    P = rs.Problem(rng.uniform(0, 1, (300, 2)), np.full(300, 1 / 300), rng.uniform(0, 1, (50, 2)),
                   np.full(50, 0.02))
    g = np.full(50, 7.0)
    try:
        for bad in (np.nan, np.inf):
            for at in (0, 17):
                psi = np.zeros(50)
                psi[at] = bad
                with pytest.raises(rs.RsotError):
                    P.eval(psi, 1e-2, 0.0, rs.FP64, grad_out=g)
                assert np.all(g == 7.0)
    finally:
        P.close()


def test_many_rows_per_thread_and_split_columns():
    """Two rows per thread and several column chunks, against the truncated FP64 passes with a
    radius just below the diameter, which keep every pair."""
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(10)
    nq, n = 70001, 9001
    x, y = rng.uniform(0.1, 0.9, (nq, 3)), rng.uniform(0.1, 0.9, (n, 3))
    x[0], y[0] = 0.0, 1.0            # the diameter's ends: the only pair cut off
    m = rng.uniform(0.5, 1.5, nq)
    nu = rng.uniform(0.5, 1.5, n)
    m, nu = m / m.sum(), nu / nu.sum()
    psi = 0.005 * rng.standard_normal(n)
    P = rs.Problem(x, m, y, nu)
    try:
        J, g, _ = P.eval(psi, 2e-3, 0.0, rs.FP64)
        J2, g2, pairs = P.eval(psi, 2e-3, np.sqrt(3.0) * (1 - 1e-9), rs.FP64)
    finally:
        P.close()
    assert pairs == nq * n - 1
    assert abs(J - J2) <= 1e-12 * abs(J2)
    # FP64 sums of up to 70,001 terms in both: 70,001 * 2^-53 = 8e-12
    assert np.max(np.abs(g - g2)) <= 2e-11 * np.max(nu)


# from 1e9 pairs on points are taken in cell order by pairs and their maxima leave out targets: an odd
# number of points in no order, against the error-free part of the compensated bound
@pytest.mark.parametrize("d,nq,n,eps", [(3, 100001, 10007, 1e-3), (2, 400003, 2503, 2e-4)])
def test_large(d, nq, n, eps):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(nq)
    x, y = rng.uniform(0, 1, (nq, d)), rng.uniform(0, 1, (n, d))
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    m, nu = m / m.sum(), nu / nu.sum()
    psi = eps * rng.standard_normal(n)
    P = rs.Problem(x, m, y, nu)
    try:
        P.kernel_timing(True)
        J, g, _ = P.eval(psi, eps, 0.0, rs.FP64)
        assert "fx_lse" in P.kernel_times()
        L = P.point_log_partition()
    finally:
        P.close()
    # every point's logarithm against a sum over all targets, for some points, and the total mass
    pick = rng.choice(nq, 200, replace=False)
    for q in pick:
        e = (psi - 0.5 * ((x[q] - y) ** 2).sum(1)) / eps + np.log(nu)
        M = e.max()
        assert abs(L[q] - (M + np.log(np.exp(e - M).sum()))) <= 1e-12 * max(1.0, abs(M))
    assert abs((g + nu).sum() - 1.0) <= 1e-12

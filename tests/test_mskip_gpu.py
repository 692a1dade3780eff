"""Mixed evaluations that leave out pairs (rsot_mskip.cu) against the FP64 evaluation.

Tolerance: the FP32 exponents' error, delta = ln2 4 2^-24 K per plan weight with K the bound of the
exponent's terms (test_maps_gpu.py), in the pair and in the normaliser; what is left out is below 2^-59 of a
sum or of nu_j.
"""
import numpy as np
import pytest

from test_maps_gpu import delta_of

pytestmark = pytest.mark.gpu


def _check(x, m, y, nu, psi, eps, forms):
    import paper_2507_23602_gb300 as rs
    P = rs.Problem(x, m, y, nu)
    try:
        J64, g64, _ = P.eval(psi, eps, 0.0, rs.FP64)
        L64 = P.point_log_partition()
        P.kernel_timing(True)
        J, g, pairs = P.eval(psi, eps, 0.0, rs.MIXED)
        names = set(P.kernel_times())
        L = P.point_log_partition()
        P.set_pair_kernel(rs.PAIRS_FP32)   # every pair: the same to 2^-59 of a sum
        Jd, gd, _ = P.eval(psi, eps, 0.0, rs.MIXED)
        Ld = P.point_log_partition()
        assert "lse_mixed" in P.kernel_times()
    finally:
        P.close()
    assert forms <= names and pairs == len(m) * len(nu)
    # FP64 sums in another order (512 points each: at most nq / 512 terms)
    order = (len(m) / 512 + 2) * 2.0 ** -52
    assert np.all(np.abs(g - gd) <= order * (gd + 2 * nu))
    assert np.all(np.abs(L - Ld) <= 2.0 ** -50 * (1 + np.abs(Ld))) and abs(J - Jd) <= 2.0 ** -50 * (1 + abs(Jd))
    rel = 2 * delta_of(x, y, nu, psi, eps) + 2.0 ** -24 * 512
    assert np.all(np.abs(g - g64) <= rel * (g64 + nu) + 1e-14 * nu)
    live = m > 0
    assert np.all(np.abs(L - L64)[live] <= rel + 1e-12 * np.abs(L64[live]))
    assert abs(J - J64) <= rel * eps + 1e-12 * abs(J64)


def _problem(d, nq, n, seed):
    rng = np.random.default_rng(seed)
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    return rng.uniform(0, 1, (nq, d)), m / m.sum(), rng.uniform(0, 1, (n, d)), nu / nu.sum(), rng


# odd numbers of points (a pair with padding) and targets, rows beyond the last whole warp, points of
# every order (the caller's is random), one chunk of targets and many
@pytest.mark.parametrize("d,nq,n,eps", [(3, 622591, 2561, 1e-3), (3, 65537, 32769, 5e-4), (2, 622590, 2600, 3e-4),
                                        (3, 2049, 800001, 5e-4), (3, 1000001, 2047, 2e-4)])
def test_sizes(d, nq, n, eps):
    x, m, y, nu, rng = _problem(d, nq, n, nq + n)
    _check(x, m, y, nu, 0.5 * eps * rng.standard_normal(n), eps, {"lse_skip", "grad_skip"})


# potentials that raise the running shifts again and again, points without mass, targets far from
# every point and points far from every target
@pytest.mark.parametrize("case", ["spread", "massless", "apart"])
def test_shifts_and_ranges(case):
    eps = 1e-3
    x, m, y, nu, rng = _problem(3, 622592, 3000, 9)
    psi = 0.5 * eps * rng.standard_normal(3000)
    if case == "spread":
        psi = 0.3 * rng.standard_normal(3000)
    if case == "massless":
        m[::3] = 0.0
    if case == "apart":
        x[:20000] += [4.0, 0.0, 0.0]
        y[:300] -= [0.0, 3.0, 0.0]
    _check(x, m / m.sum(), y, nu, psi, eps, {"lse_skip", "grad_skip"})


# the smallest work that leaves pairs out: many chunks of targets, few warps per scheduler
@pytest.mark.parametrize("d,nq,n,eps", [(3, 331777, 16383, 1e-3), (3, 98305, 16385, 1e-3), (2, 153601, 10001, 5e-4)])
def test_smaller_work(d, nq, n, eps):
    x, m, y, nu, rng = _problem(d, nq, n, nq + n)
    _check(x, m, y, nu, 0.5 * eps * rng.standard_normal(n), eps, {"lse_skip", "grad_skip"})

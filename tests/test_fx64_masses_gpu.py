"""Dense FP64 evaluations of densities and weights that reach down to the bottom of the FP64 range.

A narrow Gaussian leaves points whose mass, and with it every term m_q p_qj, lies below 2^-1022.
Tolerance: that of test_fx64_gpu.py, 1e-12 of the larger of a target's transported mass and nu_j
(1e-10 where the general FP64 passes run, whose exponents round at their own size); sums over more
than 4,096 points add 2^-53 a term.
"""
import numpy as np
import pytest

from test_fx64_gpu import LD, _exact

pytestmark = pytest.mark.gpu


def _mesh(d, cells):
    """Cell centres of the unit square's or cube's grid."""
    a = (np.arange(cells) + 0.5) / cells
    return np.stack(np.meshgrid(*[a] * d, indexing="ij"), -1).reshape(-1, d)


def _gaussian(x, sigma, at=0.2):
    """Normalised masses; the smallest are subnormal or zero (the square's far corner)."""
    m = np.exp(-0.5 * ((x - at) ** 2).sum(1) / sigma ** 2)
    return m / m.sum()


def _targets(d, n, seed):
    rng = np.random.default_rng(seed)
    nu = rng.uniform(0.5, 1.5, n)
    return rng.uniform(0, 1, (n, d)), nu / nu.sum(), 0.005 * rng.standard_normal(n)


def _eval(x, m, y, nu, psi, eps):
    import paper_2507_23602_gb300 as rs
    P = rs.Problem(x, m, y, nu)
    try:
        P.kernel_timing(True)
        J, g, _ = P.eval(psi, eps, 0.0, rs.FP64)
        return J, g, set(P.kernel_times())
    finally:
        P.close()


def _check(x, m, y, nu, psi, eps, tol=1e-12):
    J, g, names = _eval(x, m, y, nu, psi, eps)
    Je, a, L = _exact(x, m, y, nu, psi, eps)
    err = np.abs(g.astype(LD) - (a - nu.astype(LD)))
    assert np.all(err <= tol * np.maximum(a, nu)), float((err / np.maximum(a, nu)).max())
    assert abs(LD(J) - Je) <= tol * (abs(Je) + LD(eps) * np.abs(m * L).sum())
    return names


@pytest.mark.parametrize("d,cells,sigma", [(2, 30, 0.02), (2, 30, 0.025), (2, 31, 0.03), (3, 10, 0.03)])
def test_narrow_gaussian(d, cells, sigma):
    x = _mesh(d, cells)
    m = _gaussian(x, sigma)
    assert np.any((m > 0) & (m < 1e-290))
    y, nu, psi = _targets(d, 150, cells)
    assert "grad_fp64" not in _check(x, m, y, nu, psi, 1e-2)


# a few masses put where a term's exponent passes -1022 by little, by much, and in a chain of sizes
def test_masses_of_every_size():
    x = _mesh(2, 24)
    rng = np.random.default_rng(3)
    m = 10.0 ** rng.uniform(-323, 0, len(x))
    m[:40] = 5e-324
    y, nu, psi = _targets(2, 130, 4)
    _check(x, m, y, nu, psi, 1e-2)
    _check(x, m, y, nu, psi, 0.5)


# masses and weights in other units than probabilities
@pytest.mark.parametrize("scale", [1e-280, 1e-150, 1e150, 1e300])
def test_scaled_masses(scale):
    x = _mesh(2, 24)
    y, nu, psi = _targets(2, 130, 5)
    m = _gaussian(x, 0.1) * scale
    _check(x, m, y, nu, psi, 1e-2, 1e-10)
    nu = nu * scale
    _check(x, m, y, nu, psi, 1e-2, 1e-10)


# weights: ordinary passes down to about 1e-120, the general ones below
@pytest.mark.parametrize("lo,tol", [(1e-60, 1e-12), (1e-100, 1e-12), (1e-140, 1e-10), (1e-290, 1e-10),
                                    (1e-300, 1e-10)])
@pytest.mark.parametrize("sigma", [0.02, 0.3])
def test_tiny_weights(lo, tol, sigma):
    x = _mesh(2, 24)
    m = _gaussian(x, sigma)
    y, nu, psi = _targets(2, 130, 6)
    nu[::3] = lo * np.linspace(1.0, 2.0, len(nu[::3]))
    _check(x, m, y, nu, psi, 1e-2, tol)


# two rows per thread (many targets and points) and one, against the truncated FP64 passes with a radius
# just below the diameter, which keep every pair but the diameter's own
@pytest.mark.parametrize("d,cells,n", [(2, 64, 512), (2, 157, 4096), (3, 46, 1024)])
@pytest.mark.parametrize("sigma", [0.02, 0.025])
def test_against_the_general_passes(d, cells, n, sigma):
    import paper_2507_23602_gb300 as rs
    x = _mesh(d, cells)
    m = _gaussian(x, sigma)
    y, nu, psi = _targets(d, n, n)
    y[0] = 1.0                       # with x[0], the first cell's centre, nearly the diameter
    x[0] = 0.0
    P = rs.Problem(x, m, y, nu)
    try:
        J, g, _ = P.eval(psi, 1e-2, 0.0, rs.FP64)
        J2, g2, pairs = P.eval(psi, 1e-2, np.sqrt(d) * (1 - 1e-9), rs.FP64)
    finally:
        P.close()
    assert pairs == len(x) * n - 1
    assert abs(J - J2) <= 1e-12 * abs(J2)
    assert np.all(np.abs(g - g2) <= 1e-10 * (g2 + 2 * nu))


def test_solve_in_fp64():
    import paper_2507_23602_gb300 as rs
    x = _mesh(2, 64)
    m = _gaussian(x, 0.025)
    y, nu, _ = _targets(2, 512, 7)
    P = rs.Problem(x, m, y, nu)
    try:
        psi, st = P.solve(eps=2e-2, tol_l1=1e-6, precision=rs.FP64)
        _, g, _ = P.eval(psi, 2e-2, np.sqrt(2.0) * 0.999, rs.FP64)   # the general passes
    finally:
        P.close()
    assert st.status == 0 and np.abs(g).sum() <= 1e-6 + 1e-10

"""Two handles of the same data give the same bits: the orders that a handle makes for its rows depend on the
data alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# many rows to a cell, clustered rows (most in few cells), an odd number of points
@pytest.mark.parametrize("d,nq,n,eps,clustered", [(3, 98305, 16385, 1e-3, False), (2, 200001, 9001, 5e-4, False),
                                                  (3, 98305, 16385, 1e-3, True)])
def test_same_bits(d, nq, n, eps, clustered):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(nq)
    x, y = rng.uniform(0, 1, (nq, d)), rng.uniform(0, 1, (n, d))
    if clustered:
        y[: n - 100] = 0.5 + 0.02 * rng.standard_normal((n - 100, d))
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    m, nu = m / m.sum(), nu / nu.sum()
    psi = eps * rng.standard_normal(n)
    results = []
    for order in ("fp64 first", "mixed first", "again"):
        P = rs.Problem(x, m, y, nu)
        try:
            if order == "mixed first":
                P.eval(psi, eps, 0.0, rs.MIXED)
            out = []
            for prec in (rs.FP64, rs.MIXED, rs.COMPENSATED):
                J, g, _ = P.eval(psi, eps, 0.0, prec)
                out += [J, g, P.point_log_partition()]
        finally:
            P.close()
        results.append(out)
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert np.array_equal(a, b), int(np.sum(np.asarray(a) != np.asarray(b)))

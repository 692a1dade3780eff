"""Evaluations of few points against many targets, around the sizes where a pass may start before the kernel
in front of it has ended (points' CTAs and targets' blocks against the number of SMs) and where the points'
maxima and the compensated pass take one tile of targets per CTA.

Tolerances: FP64 1e-12 of the larger of a target's transported mass and nu_j (exponents below 160 here, a
rounding of 2^-53 each in the sums formed on the host); mixed 3e-5 (test_eval_tail_gpu.py); compensated its
bound of 6.0e-7.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,nq,n", [(2, 16, 1000), (3, 64, 1024), (2, 300, 1025), (3, 1024, 2047), (2, 1025, 4096),
                                    (2, 16, 4097), (3, 1536, 8000), (2, 3000, 8193), (2, 16, 16000), (3, 300, 30000),
                                    (3, 6000, 128), (2, 6145, 257)])
def test_every_precision(d, nq, n):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(nq + n)
    eps = 1e-2
    x, y = rng.uniform(0, 1, (nq, d)), rng.uniform(0, 1, (n, d))
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    m, nu = m / m.sum(), nu / nu.sum()
    psi = 0.005 * rng.standard_normal(n)
    a, J = np.zeros(n), -(psi * nu).sum()
    for q in range(0, nq, 256):
        s = (psi - 0.5 * ((x[q:q + 256, None] - y[None]) ** 2).sum(-1)) / eps + np.log(nu)
        top = s.max(1)
        p = np.exp(s - top[:, None])
        S = p.sum(1)
        J += (m[q:q + 256] * eps * (top + np.log(S))).sum()
        a += (m[q:q + 256] / S) @ p
    P = rs.Problem(x, m, y, nu)
    try:
        got = {k: P.eval(psi, eps, 0.0, getattr(rs, k)) for k in ("FP64", "MIXED", "COMPENSATED")}
        T, mass = P.centroids(psi, eps)
    finally:
        P.close()
    for k, tol in (("FP64", 1e-12), ("MIXED", 3e-5), ("COMPENSATED", 6.0e-7)):
        Jk, g, _ = got[k]
        assert np.all(np.abs(g + nu - a) <= tol * a + 1e-12 * nu), k
        assert abs(Jk - J) <= max(1e-12, tol * eps), k
    assert np.all(np.abs(mass - a) <= 3e-5 * a + 1e-12 * nu)

"""The last kernel of an evaluation (rsot_dense.cu, k_finalize) and pass 2's split of small problems.

Every form that ends with that kernel, with host, device and overlapping buffers, after an error
and after a truncated evaluation: the results of one problem are the same bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(d, nq, n, seed=3):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(seed)
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    return (rs, rs.Problem(rng.uniform(0, 1, (nq, d)), m / m.sum(), rng.uniform(0, 1, (n, d)), nu / nu.sum()),
            0.01 * rng.standard_normal(n), nu / nu.sum())


@pytest.mark.parametrize("prec", ["FP64", "MIXED", "COMPENSATED"])
@pytest.mark.parametrize("d,nq,n", [(2, 1, 1), (3, 257, 255), (2, 1500, 1025), (2, 80000, 300)])
def test_buffers_and_errors(d, nq, n, prec):
    import torch
    rs, P, psi, _ = _problem(d, nq, n)
    prec = getattr(rs, prec)
    try:
        J, g, _ = P.eval(psi, 1e-2, 0.0, prec)
        dev = torch.tensor(psi, device="cuda")
        Jd, gd, _ = P.eval(dev, 1e-2, 0.0, prec)
        assert Jd == J and np.array_equal(gd.cpu().numpy(), g)
        Jo, go, _ = P.eval(dev, 1e-2, 0.0, prec, grad_out=dev)   # the gradient over the potential
        assert Jo == J and np.array_equal(go.cpu().numpy(), g)
        bad = psi.copy()
        bad[n // 2] = np.nan
        out = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
        with pytest.raises(rs.RsotError):
            P.eval(torch.tensor(bad, device="cuda"), 1e-2, 0.0, prec, grad_out=out)
        assert bool((out == 7.0).all())
        for radius in (0.0, 0.3, 0.0):   # after an error, and after a truncated evaluation
            try:
                Ja, ga, pairs = P.eval(psi, 1e-2, radius, prec)
            except rs.RsotError:
                continue
            if radius == 0.0:
                assert Ja == J and np.array_equal(ga, g) and pairs == nq * n
    finally:
        P.close()


def test_empty_neighbourhood_writes_nothing():
    import torch
    rs, P, psi, _ = _problem(2, 700, 40)
    try:
        for prec in (rs.FP64, rs.MIXED, rs.COMPENSATED):
            out = torch.full((40,), 7.0, dtype=torch.float64, device="cuda")
            with pytest.raises(rs.RsotError):
                P.eval(torch.tensor(psi, device="cuda"), 1e-2, 0.02, prec, grad_out=out)
            assert bool((out == 7.0).all())
            assert P.last_eval()[3] > 0
    finally:
        P.close()


# around 64 stages of 512 points and around one wave of CTAs, where the split changes.  The mixed
# evaluation's gradient terms err by less than 1e-5 of a target's mass here (exponents up to ~ 150
# in FP32 fused multiply-adds of rounded operands: (150 + 4) 2^-23 ln 2 in pass 1 and in pass 2)
@pytest.mark.parametrize("d,nq,n", [(2, 511, 7), (3, 513, 700), (2, 32768, 300), (2, 32769, 300),
                                    (2, 9600, 24000)])
def test_split_of_small_problems(d, nq, n):
    rs, P, psi, nu = _problem(d, nq, n)
    try:
        J64, g64, _ = P.eval(psi, 1e-2, 0.0, rs.FP64)
        J, g, _ = P.eval(psi, 1e-2, 0.0, rs.MIXED)
    finally:
        P.close()
    assert abs(J - J64) <= 1e-6 * 1e-2 * 154 + 1e-12
    assert np.all(np.abs(g - g64) <= 3e-5 * (g64 + nu))


# host potentials of at most 65,536 entries are read in place by the target records' kernel
@pytest.mark.parametrize("prec", ["FP64", "MIXED", "COMPENSATED"])
@pytest.mark.parametrize("n", [65536, 65537])
def test_host_potential_read_or_copied(n, prec):
    import torch
    rs, P, psi, _ = _problem(3, 64, n)
    try:
        for k in range(2):
            psi = psi + 0.001 * k
            J, g, _ = P.eval(psi, 1e-2, 0.0, getattr(rs, prec))
            Jd, gd, _ = P.eval(torch.tensor(psi, device="cuda"), 1e-2, 0.0, getattr(rs, prec))
            assert J == Jd and np.array_equal(g, gd.cpu().numpy())
    finally:
        P.close()

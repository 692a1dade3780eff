"""Dense evaluations after failed and truncated ones: the result block that the last kernel clears
(rsot_dense.cu, k_finalize) carries nothing over."""
import numpy as np
import pytest

from test_result_block_gpu import _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP64", "MIXED", "COMPENSATED"])
@pytest.mark.parametrize("d,nq,n", [(2, 1, 1), (3, 257, 255), (2, 1500, 1025), (2, 80000, 300)])
def test_dense_evaluations_after_errors(d, nq, n, prec):
    """Dense evaluations return the same bits directly after a refused potential, after a truncated
    evaluation (whose points may have no target) and after a refinement."""
    rs, P, psi = _problem(d, nq, n)
    prec = getattr(rs, prec)
    try:
        J, g, _ = P.eval(psi, 1e-2, 0.0, prec)

        def same():
            Ja, ga, pairs = P.eval(psi, 1e-2, 0.0, prec)
            assert Ja == J and np.array_equal(ga, g) and pairs == nq * n

        bad = psi.copy()
        bad[n // 2] = np.nan
        for other in (rs.FP64, rs.MIXED, rs.COMPENSATED):
            with pytest.raises(rs.RsotError):
                P.eval(bad, 1e-2, 0.0, other)
            same()
            try:
                P.eval(psi, 1e-2, 0.3, other)
            except rs.RsotError as e:
                assert e.status == rs.RSOT_ERR_EMPTY_NEIGHBORHOOD
            same()
        with pytest.raises(rs.RsotError):
            P.softmax_refine(bad, 1e-2, np.zeros((3, d)))
        same()
    finally:
        P.close()

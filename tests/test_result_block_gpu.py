"""The result block that the last kernel of an evaluation clears (rsot_dense.cu, k_finalize)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(d, nq, n, seed=3):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(seed)
    m, nu = rng.uniform(0.2, 1.8, nq), rng.uniform(0.5, 1.5, n)
    return (rs, rs.Problem(rng.uniform(0, 1, (nq, d)), m / m.sum(), rng.uniform(0, 1, (n, d)), nu / nu.sum()),
            0.01 * rng.standard_normal(n))


@pytest.mark.parametrize("tensor", [False, True])
def test_centroid_sums_precede_the_last_kernel(tensor):
    """What the centroids' pass reports (a wait that ran out) is part of the evaluation's result: the last
    kernel, which hands the flags to the host and clears them, runs after it."""
    rs, P, psi = _problem(2, 600, 300)
    try:
        P.set_pair_kernel(rs.PAIRS_TENSOR if tensor else rs.PAIRS_AUTO)
        P.kernel_timing(True)
        P.centroids(psi, 1e-2)
        names = list(P.kernel_times())   # in the order of their first launch
    finally:
        P.close()
    assert ("grad_tc" in names) == tensor
    assert names.index("grad_centroids") < names.index("finalize") < names.index("centroids")

"""A potential in pinned host memory is read in stream order: what earlier work on the handle's stream writes
there is what the evaluation sees."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP64", "MIXED", "COMPENSATED"])
@pytest.mark.parametrize("n,radius", [(1500, 0.0), (1500, 0.9), (70000, 0.0)])
def test_read_after_earlier_work(n, radius, prec):
    import torch
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(n)
    nq, prec = 300, getattr(rs, prec)
    nu = rng.uniform(0.5, 1.5, n)
    P = rs.Problem(rng.uniform(0, 1, (nq, 2)), np.full(nq, 1 / nq), rng.uniform(0, 1, (n, 2)), nu / nu.sum())
    try:
        psi = 0.01 * rng.standard_normal(n)
        J, g, _ = P.eval(psi, 1e-2, radius, prec)
        dev = torch.tensor(psi, device="cuda")
        pin = torch.zeros(n, dtype=torch.float64).pin_memory()
        torch.cuda._sleep(100_000_000)   # about 50 ms of earlier work
        pin.copy_(dev, non_blocking=True)
        Jp, gp, _ = P.eval(pin, 1e-2, radius, prec)
    finally:
        P.close()
    assert Jp == J and np.array_equal(np.asarray(gp), g)

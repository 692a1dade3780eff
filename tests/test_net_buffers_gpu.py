"""The network's buffers grow apart: those of the rows, and the pinned one of forward calls whose results go
to host memory.  Every order of calls gives the results of a fresh handle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [64, 96, 256])
def test_calls_of_growing_and_shrinking_sizes(width):
    import torch
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(1)
    x = rng.normal(0, 1, (9001, 3)).astype(np.float32)
    y = rng.normal(0, 1, 9001).astype(np.float32)

    def fresh(rows):
        net = rs.MLP(3, width, seed=2)
        try:
            return net.forward(x[:rows]), net.gradients(x[:rows], y[:rows])
        finally:
            net.close()

    want = {rows: fresh(rows) for rows in (1, 128, 129, 5000, 9001)}
    net = rs.MLP(3, width, seed=2)
    try:
        for call, rows in (("f", 128), ("g", 5000), ("f", 129), ("d", 9001), ("f", 5000), ("f", 9001), ("g", 1),
                           ("f", 1), ("d", 128), ("f", 9001)):
            o, (loss, g) = want[rows]
            if call == "g":
                l2, g2 = net.gradients(x[:rows], y[:rows])
                assert l2 == loss and np.array_equal(g2, g)
            elif call == "d":
                out = net.forward(torch.tensor(x[:rows], device="cuda"), out=torch.empty(rows, device="cuda"))
                assert np.array_equal(out.cpu().numpy(), o)
            else:
                assert np.array_equal(net.forward(x[:rows]), o)
    finally:
        net.close()

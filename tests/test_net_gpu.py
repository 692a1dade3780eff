"""The network in one kernel (rsot_mlp.cu, k_net) at the edges of its tiles, and its input and output
buffers.  It does a row's arithmetic and sums in the order of the per-layer kernels, so the cp.async
form of those gives the same bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _net(in_dim, width, rows, seed=5):
    import paper_2507_23602_gb300 as rs
    rng = np.random.default_rng(seed)
    return (rs, rs.MLP(in_dim, width, seed=seed), rng.normal(0, 1, (rows, in_dim)).astype(np.float32),
            rng.normal(0, 1, rows).astype(np.float32))


# one row, a warp's rows and one more or less, a tile's; widths of one to four 64-column blocks; one
# and two 32-column input blocks; 32-, 64- and 128-row tiles on 152 SMs, one and two CTAs per SM and
# more than one tile per CTA
@pytest.mark.parametrize("in_dim,width,rows", [(1, 64, 1), (18, 256, 31), (32, 128, 33), (33, 192, 127),
                                               (64, 256, 129), (18, 192, 4865), (5, 256, 9729),
                                               (18, 256, 19457), (18, 64, 40000), (18, 256, 65535)])
def test_equal_to_the_layer_kernels(in_dim, width, rows):
    rs, net, x, y = _net(in_dim, width, rows)
    try:
        o, (l, g) = net.forward(x), net.gradients(x, y)
        net.set_gemm_kernel(rs.GEMM_TCGEN05_CPASYNC)
        o2, (l2, g2) = net.forward(x), net.gradients(x, y)
    finally:
        net.close()
    assert np.array_equal(o, o2) and l == l2 and np.array_equal(g, g2)
    assert np.all(np.isfinite(o)) and np.all(np.isfinite(g)) and np.abs(g).max() > 0


def test_buffers():
    import torch
    rs, net, x, y = _net(1, 64, 700)
    try:
        o, (l, g) = net.forward(x), net.gradients(x, y)
        xd, yd = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
        od = net.forward(xd, out=torch.empty(700, device="cuda"))
        assert np.array_equal(od.cpu().numpy(), o) and np.array_equal(net.forward(xd), o)
        ld, gd = net.gradients(xd, yd)
        assert ld == l and np.array_equal(gd, g)
        pin = torch.tensor(x).pin_memory()
        assert np.array_equal(net.forward(pin, out=torch.empty(700).pin_memory()).numpy(), o)
        odd = np.zeros(4 * 700 + 1, dtype=np.uint8)[1:].view(np.float32)   # not on a 4-byte boundary
        odd[:] = x[:, 0]
        assert np.array_equal(net.forward(odd.reshape(700, 1)), o)
        net.forward(xd, out=xd)   # the results over the input
        assert np.array_equal(xd.cpu().numpy()[:, 0], o)
    finally:
        net.close()


def test_extreme_preactivations():
    """SiLU and its derivative far from zero: exp(-z) overflows or vanishes."""
    rs, net, x, y = _net(2, 64, 64)
    try:
        p = np.zeros(net.n_params, dtype=np.float32)
        p[64 * 32:64 * 32 + 64] = np.repeat([-3e4, -200.0, -90.0, -20.0, 20.0, 90.0, 200.0, 3e4], 8)   # b1
        at = 64 * 32 + 64
        p[at:at + 64 * 64] = np.eye(64).ravel()                                     # W2
        p[at + 64 * 64 + 64:at + 2 * 64 * 64 + 64] = np.eye(64).ravel()             # W3
        p[at + 2 * (64 * 64 + 64):at + 2 * (64 * 64 + 64) + 64] = 1.0 / 64          # w4
        net.set_params(p)
        o, (l, g) = net.forward(x), net.gradients(x, y)
    finally:
        net.close()
    silu = lambda z: z / (1 + np.exp(-np.clip(z, -700, 700)))
    bf = lambda v: (np.asarray(v, np.float32).view(np.uint32) + 0x8000 & 0xFFFF0000).view(np.float32)
    h = p[64 * 32:64 * 32 + 64].astype(np.float64)
    for _ in range(3):
        h = bf(silu(h)).astype(np.float64)
    # BF16 roundings (2^-9 each, those of h to even or up at a tie) and FP32 sums
    assert np.all(np.abs(o - h.sum() / 64) <= 2.0 ** -8 * np.abs(h).sum() / 64)
    assert np.isfinite(l) and np.all(np.isfinite(g))

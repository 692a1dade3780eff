"""Centroids from pass 2 (rsot_dense.cu, k_grad_mixed with CENT) and the two-point maps (rsot_maps.cu)
at the edges of their stages, halves, sub-tiles and blocks, against the oracle.

Tolerances as in test_maps_gpu.py: delta = ln2 4 2^-24 K per plan weight, K the bound of the
exponent's terms; a_j and nu_j T_j err by at most (delta of the pair + delta of the normaliser) of
the transported mass, plus 2^-24 256 for the FP32 sums.
"""
import numpy as np
import pytest

import oracle
from test_maps_gpu import case, delta_of

pytestmark = pytest.mark.gpu

SIZES = [(2, 1, 1), (3, 255, 15), (2, 256, 17), (3, 257, 255), (2, 511, 256), (3, 513, 513), (2, 1025, 1025),
         (3, 70000, 300), (2, 4097, 1500)]


def _run(d, nq, n, tensor=False):
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, psi, eps = case(nq + n, d, nq, n, 0.02, 0.02)
    P = rs.Problem(x, m, y, nu)
    try:
        if tensor:
            P.set_pair_kernel(rs.PAIRS_TENSOR)
        T, a = P.centroids(psi, eps)
        g = P.last_eval()[1]
        Tb, js = P.transport_maps(psi, eps)
    finally:
        P.close()
    return x, m, y, nu, psi, eps, T, a, g, Tb, js


def _plan(x, m, y, nu, psi, eps):
    c = 0.5 * ((x[:, None, :] - y[None, :, :]) ** 2).sum(-1)
    r = (psi[None, :] - c) / eps + np.log(nu)[None, :]
    p = np.exp(r - r.max(1, keepdims=True))
    return r, p / p.sum(1, keepdims=True)


@pytest.mark.parametrize("tensor", [False, True])
@pytest.mark.parametrize("d,nq,n", SIZES)
def test_sums(d, nq, n, tensor):
    x, m, y, nu, psi, eps, T, a, g, Tb, js = _run(d, nq, n, tensor)
    r, p = _plan(x, m, y, nu, psi, eps)
    # the tensor-core exponents err by about twice the FP32 chain's
    rel = (2 if not tensor else 6) * delta_of(x, y, nu, psi, eps) + 2.0 ** -24 * 256
    ao = m @ p
    To = (m[:, None] * p).T @ x / nu[:, None]
    assert np.all(np.abs(a - ao) <= rel * ao + 1e-14)
    assert np.all(np.abs(T - To) * nu[:, None] <= rel * ao[:, None] * np.abs(x).max() + 1e-14)
    assert np.all(np.abs(g - (ao - nu)) <= rel * ao + 1e-14)
    assert np.all(np.abs(Tb - p @ y) <= 2 * rel * 2.0)
    jo = r.argmax(1)
    rows = np.arange(nq)
    assert np.all(r[rows, js] >= r[rows, jo] - 2 * delta_of(x, y, nu, psi, eps) * (1 + 2 * tensor))


def test_failed_evaluation_writes_nothing_and_buffers():
    import torch
    import paper_2507_23602_gb300 as rs
    x, m, y, nu, psi, eps = case(3, 2, 600, 70, 0.02, 0.02)
    P = rs.Problem(x, m, y, nu)
    try:
        T, a = P.centroids(psi, eps)
        bad = psi.copy()
        bad[3] = np.inf
        lib, out = rs.load(), torch.full((70, 2), 7.0, dtype=torch.float64, device="cuda")
        b = torch.tensor(bad, device="cuda")
        assert lib.rsot_centroids(P._h, b.data_ptr(), eps, out.data_ptr(), None) != 0
        assert bool((out == 7.0).all())
        g = torch.tensor(psi, device="cuda")
        assert lib.rsot_centroids(P._h, g.data_ptr(), eps, out.data_ptr(), None) == 0
        assert np.array_equal(out.cpu().numpy(), T)
        assert oracle is not None
    finally:
        P.close()

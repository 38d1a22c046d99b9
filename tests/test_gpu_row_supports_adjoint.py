"""Dense adjoint where pairs and G vectors live on different terms of the products
(see test_gpu_row_supports.py for the bar): every gradient element is held to its own S."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BAR = 2.0 ** -49


@pytest.mark.parametrize("nG,K,t,max_pairs,precision", [
    (70, 90, 1e-6, 0, "fp64"), (150, 300, 1e-9, 128, "fp64"), (257, 64, 1e-3, 0, "fp64"), (129, 200, 1e-9, 0, "fp16"),
])
def test_adjoint_rows_on_different_terms(nG, K, t, max_pairs, precision):
    """f = f' = -1: gM = -(M G^T + M conj(G)), grad dE = -Re sum conj(M) (M G^T)."""
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    rng = np.random.default_rng(nG)
    dt = np.complex128 if precision == "fp64" else np.complex64
    half = rng.permutation(nG) < nG // 2
    M = rng.standard_normal((K, nG)) + 1j * rng.standard_normal((K, nG))
    G = rng.standard_normal((nG, nG)) + 1j * rng.standard_normal((nG, nG))
    M = np.where(half[None] == (rng.integers(0, 2, K) > 0)[:, None], M, t * M).astype(dt)
    G = np.where(half[None] == half[:, None], G, t * G)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], [0.0], 0.0, precision=precision, max_pairs=max_pairs) as plan:
        gM, gv, gc = plan.backward(0, dev(M), 1, K, dev(np.zeros(1)), dev(np.ones(K)), grad_chi=dev(G[None]))
        plan.sync_status()
    M = M.astype(np.complex128)
    Y, Z, S = M @ G.T, M @ G.conj(), np.abs(M) @ (np.abs(G) + np.abs(G.T)).T
    bar = BAR * S if precision == "fp64" else 2.0 ** -23 * np.abs(Y + Z) + BAR * S
    assert np.all(np.abs(gM.cpu().numpy() + Y + Z) <= bar)
    dE = -(M.conj() * Y).sum(1).real
    assert np.all(np.abs(gc.cpu().numpy() + dE) <= BAR * (np.abs(M) * S).sum(1))

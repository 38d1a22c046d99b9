"""The diagonal adjoint where its grouping of pairs, its reductions and its range
checks end: pair counts that are no multiple of four, rows and columns cut by the
pair blocks, one and several frequencies, gradients g outside the FP32 range.

Energies: FP64 sums of positive terms, 1e-14.  complex64 gradients: one rounding
(2^-24 of each value, the bar 2^-24 in the Frobenius norm); complex128 1e-14."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp16"])
@pytest.mark.parametrize("nG,n_v,n_c,n_freq,max_pairs,g_scale", [
    (1, 1, 1, 1, 0, 1.0), (2, 3, 7, 1, 0, 1.0), (33, 1, 203, 1, 64, 1.0), (129, 70, 1, 1, 64, 1.0),
    (57, 5, 41, 2, 128, 1.0), (350, 9, 33, 3, 64, 1.0), (130, 4, 9, 1, 0, 2.0 ** 41), (130, 4, 9, 1, 0, 2.0 ** -45),
])
def test_diagonal_adjoint_edges(nG, n_v, n_c, n_freq, max_pairs, g_scale, precision):
    import torch
    from oracle import chi0_grad
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    rng = np.random.default_rng(nG + n_v)
    K = n_v * n_c
    cdt = np.complex128 if precision == "fp64" else np.complex64
    M = (rng.standard_normal((K, nG)) + 1j * rng.standard_normal((K, nG))).astype(cdt)
    Ev, Ec, w = -rng.uniform(0, 0.25, n_v), rng.uniform(0.2, 2.0, n_c), rng.uniform(0.5, 2.0, n_c)
    omega = np.concatenate([[0.0], 0.3j * np.arange(1, n_freq)])
    g = rng.uniform(0.0, 1.0, (n_freq, nG)) * g_scale
    g[0, 0] = 0.0
    dE = (Ev[:, None] - Ec[None]).reshape(-1)
    rM, rd = chi0_grad(M.astype(complex), dE, np.tile(w, n_v), omega, 1e-3, np.stack([np.diag(x) for x in g]).astype(complex))
    rd = rd.reshape(n_v, n_c)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], omega, 1e-3, precision=precision, max_pairs=max_pairs) as plan:
        gM, gEv, gEc = plan.backward(0, dev(M), n_v, n_c, dev(Ev), dev(Ec), dev(w), diag_g=dev(g))
        plan.sync_status()
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / (np.linalg.norm(b) or 1.0)
    assert rel(gM, rM) < (1e-14 if precision == "fp64" else 2.0 ** -24)
    assert rel(gEv, rd.sum(1)) < 1e-14 and rel(gEc, -rd.sum(0)) < 1e-14


def test_diagonal_adjoint_infinities():
    """An infinite pair element gives an infinite gradient, not a NaN, also where the factor's low part is zero."""
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    M = torch.ones((5, 16), dtype=torch.complex64, device="cuda")
    M[2, 3] = complex(float("inf"), 1.0)
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    with Chi0Plan(24, [g_sphere(16, (0.0, 0.0, 0.0))], [0.0], 0.0, precision="fp16") as plan:
        gM, gEv, _ = plan.backward(0, M, 1, 5, 0 * one, torch.ones(5, dtype=torch.float64, device="cuda"),
                                   diag_g=torch.ones((1, 16), dtype=torch.float64, device="cuda"))
    gM = gM.cpu().numpy()
    assert gM[2, 3].real == -np.inf and gM[2, 3].imag == -2.0
    assert np.isfinite(np.delete(gM.ravel(), 2 * 16 + 3)).all() and np.isinf(gEv.cpu().numpy()).all()

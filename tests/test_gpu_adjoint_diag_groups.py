"""The diagonal adjoint around the pair count where a CTA changes from one pair to four
(912), the last group full and cut, one and several frequencies.

Bars as in test_gpu_adjoint_diag.py: energies 1e-14, complex64 gradients one
rounding (2^-24), complex128 1e-14."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp16"])
@pytest.mark.parametrize("nG,n_v,n_c,n_freq", [(33, 8, 114, 1), (33, 11, 83, 1), (129, 83, 11, 3), (57, 7, 172, 5), (300, 1, 1202, 1)])
def test_group_sizes(nG, n_v, n_c, n_freq, precision):
    import torch
    from oracle import chi0_grad
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    rng = np.random.default_rng(nG + n_v)
    K = n_v * n_c
    M = (rng.standard_normal((K, nG)) + 1j * rng.standard_normal((K, nG))).astype(np.complex128 if precision == "fp64" else np.complex64)
    Ev, Ec = -rng.uniform(0, 0.25, n_v), rng.uniform(0.2, 2.0, n_c)
    omega = np.concatenate([[0.0], 0.3j * np.arange(1, n_freq)])
    g = rng.uniform(0.0, 1.0, (n_freq, nG))
    dE = (Ev[:, None] - Ec[None]).reshape(-1)
    rM, rd = chi0_grad(M.astype(complex), dE, np.ones(K), omega, 1e-3, np.stack([np.diag(x) for x in g]).astype(complex))
    rd = rd.reshape(n_v, n_c)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], omega, 1e-3, precision=precision) as plan:
        gM, gEv, gEc = plan.backward(0, dev(M), n_v, n_c, dev(Ev), dev(Ec), diag_g=dev(g))
        plan.sync_status()
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    assert rel(gM, rM) < (1e-14 if precision == "fp64" else 2.0 ** -24)
    assert rel(gEv, rd.sum(1)) < 1e-14 and rel(gEc, -rd.sum(0)) < 1e-14

"""Pair blocks longer than 65535 rows of CTAs: a handful of G vectors with millions of
pairs in one block (max_pairs), FP64 contraction and dense adjoint."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _plan(nG, K):
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    return Chi0Plan(8, [g_sphere(nG, (0.0, 0.0, 0.0))], [0.0], 0.0, precision="fp64", max_pairs=K)


def test_contraction_of_four_million_pairs():
    """Integers: exact on every route."""
    import torch
    nG, K = 3, 65535 * 64 + 200
    M = torch.randint(-9, 10, (K, nG, 2), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    M = torch.view_as_complex(M.double())
    with _plan(nG, K) as plan:
        chi = plan.accumulate(0, M, 1, K, torch.zeros(1, device="cuda", dtype=torch.float64),
                              torch.ones(K, device="cuda", dtype=torch.float64))
        plan.sync_status()
    assert torch.equal(chi[0], -(M.T @ M.conj()))


def test_dense_adjoint_of_a_million_pairs():
    """f = -1 and f' = -1: gM = -(M G^T + M conj(G)), grad dE = -Re sum conj(M) (M G^T); FP64 sums of 8 terms, 1e-14.
    All pairs lie in one row, whose sum of 1e6 terms is held to 1e-12 of their magnitudes."""
    import torch
    nG, K = 8, 65535 * 16 + 100
    gen = torch.Generator("cuda").manual_seed(2)
    M = torch.view_as_complex(torch.randn((K, nG, 2), device="cuda", dtype=torch.float64, generator=gen))
    G = torch.view_as_complex(torch.randn((1, nG, nG, 2), device="cuda", dtype=torch.float64, generator=gen))
    with _plan(nG, K) as plan:
        gM, gv, gc = plan.backward(0, M, 1, K, torch.zeros(1, device="cuda", dtype=torch.float64),
                                   torch.ones(K, device="cuda", dtype=torch.float64), grad_chi=G)
        plan.sync_status()
    Y = M @ G[0].T
    ref, dE = -(Y + M @ G[0].conj()), -(M.conj() * Y).sum(1).real
    rel = lambda a, b: float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))
    assert rel(gM, ref) < 1e-14 and rel(gc, -dE) < 1e-14
    assert abs(float(gv[0] - dE.sum())) < 1e-12 * float(dE.abs().sum())

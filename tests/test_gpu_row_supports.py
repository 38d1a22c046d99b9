"""FP64 contraction and dense adjoint where the rows of a product live on different
terms, so that S = sum |a||b| is far below the product of their norms: the error
of each element is held to its own S.

A sequential FP64 sum of K terms of random phase carries about 0.2 x 2^-53 of S, the
modular products at most 0.08 x 32 x 2^-53 of it where they run, the reference
as much as the former: 2^-49 of S is 16 x 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BAR = 2.0 ** -49


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _plan(nG, omega, delta, **kw):
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    return Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], omega, delta, precision="fp64", **kw)


def _complex(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _damp(rng, x, t):
    """Every row of x keeps one of two halves of its terms and has the other times t."""
    half = rng.integers(0, 2, x.shape[0])[:, None] == (rng.permutation(x.shape[1]) < x.shape[1] // 2)[None]
    return np.where(half, x, t * x)


def _held(got, ref, S):
    assert np.all(np.abs(got - ref) <= BAR * S), float(np.max(np.abs(got - ref)[S > 0] / S[S > 0]) * 2.0 ** 53)


@pytest.mark.parametrize("nG,K,t,n_freq", [(70, 2048, 1e-6, 1), (130, 700, 1e-9, 2), (300, 512, 1e-3, 1), (65, 3000, 0.0, 1)])
def test_contraction_rows_on_different_pairs(nG, K, t, n_freq):
    rng = np.random.default_rng(nG)
    M = _damp(rng, _complex(rng, nG, K), t).T
    with _plan(nG, np.zeros(n_freq), 0.0) as plan:                        # f = -1
        chi = plan.accumulate(0, _dev(M), 1, K, _dev(np.zeros(1)), _dev(np.ones(K))).cpu().numpy()
        plan.sync_status()
    ref, S = -(M.T @ M.conj()), np.abs(M).T @ np.abs(M)
    for c in chi:
        _held(c, ref, S)


def test_contraction_some_rows_only():
    """One pair of rows out of 400 apart: its tile alone takes the other route, at both sides of the diagonal."""
    rng = np.random.default_rng(2)
    nG, K = 400, 600
    M = _complex(rng, K, nG)
    M[:K // 2, 7] *= 1e-8
    M[K // 2:, 390] *= 1e-8
    with _plan(nG, [0.0], 0.0) as plan:
        chi = plan.accumulate(0, _dev(M), 1, K, _dev(np.zeros(1)), _dev(np.ones(K))).cpu().numpy()[0]
        plan.sync_status()
    _held(chi, -(M.T @ M.conj()), np.abs(M).T @ np.abs(M))


def test_contraction_resonant_factor():
    """One pair within 1e-9 of a pole: its factor outweighs the others by 1e8 at that frequency alone.
    (Reference in extended precision: a chain of FP64 sums rounds K times at the size of the one term.)"""
    rng = np.random.default_rng(3)
    nG, K, delta = 100, 500, 1e-9
    M, E = _complex(rng, K, nG), rng.uniform(0.2, 2.0, K)
    omega = np.array([0.0, E[17] + 1e-9])
    with _plan(nG, omega, delta) as plan:
        chi = plan.accumulate(0, _dev(M), 1, K, _dev(np.zeros(1)), _dev(E)).cpu().numpy()
        plan.sync_status()
    L, EL = M.astype(np.clongdouble), E.astype(np.longdouble)
    for c, om in zip(chi, omega):
        f = sum(1 / (x + np.clongdouble(1j * delta)) for x in (-EL - np.longdouble(om), -EL + np.longdouble(om))) / 2
        ref = (f[:, None] * L).T @ L.conj()
        _held(c, ref, (np.abs(f[:, None] * L).T @ np.abs(L)).astype(float))

"""The refined FP64 inverse (FP32 elimination and modular Newton steps) where it
begins, where it gives way to the FP64 elimination, and next to such matrices.

Well-conditioned matrices: 1e-13 x cond as in the other FP64 inverse tests.  Where
a matrix is ill conditioned for FP32, outside FP32's range or singular, the FP64
elimination's answer is expected: the same bar, non-finite values, or the status."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _inverse(E):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    with Chi0Plan(24, [g_sphere(E.shape[-1], (0.0, 0.0, 0.0))], np.zeros(len(E)), 1e-3, precision="fp64") as plan:
        t = plan.epsilon_inverse(0, torch.from_numpy(E.copy()).cuda())
        status = None
        try:
            plan.sync_status()
        except Exception as exc:
            status = exc
        return t.cpu().numpy(), status


def _matrix(rng, n, cond=None, scale=1.0):
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if cond is None:
        return scale * (np.eye(n) + 0.4 * A / np.sqrt(n))
    u, _, v = np.linalg.svd(A)
    return scale * (u * np.logspace(0, -np.log10(cond), n)) @ v


@pytest.mark.parametrize("n", [63, 64, 65, 127, 130, 256, 257, 321])
def test_refined_sizes(n):
    rng = np.random.default_rng(n)
    E = np.stack([_matrix(rng, n), _matrix(rng, n, cond=300.0)])
    got, status = _inverse(E)
    assert status is None
    for g, e in zip(got, E):
        r = np.linalg.inv(e)
        assert np.linalg.norm(g - r) / np.linalg.norm(r) < 1e-13 * np.linalg.cond(e)


def test_mixed_matrices_fall_back_alone():
    rng = np.random.default_rng(9)
    n = 96
    E = np.stack([_matrix(rng, n), _matrix(rng, n, cond=1e9), _matrix(rng, n, scale=1e150), _matrix(rng, n, scale=1e-60),
                  _matrix(rng, n)])
    got, status = _inverse(E)
    assert status is None
    for g, e in zip(got, E):
        s = np.abs(e).max()
        r = np.linalg.inv(e / s) / s
        assert np.linalg.norm(g * s - r * s) / np.linalg.norm(r * s) < 1e-13 * np.linalg.cond(e / s)


def test_singular_and_nonfinite_matrices_beside_good_ones():
    import paper_1601_06767_gb300._lib as L
    rng = np.random.default_rng(10)
    n = 80
    E = np.stack([_matrix(rng, n) for _ in range(4)])
    E[1, :, 7] = 0.0
    E[3, 5, 6] = np.nan
    got, status = _inverse(E)
    assert status is not None and status.status == L.CHI0_ERR_SINGULAR
    for i in (0, 2):
        r = np.linalg.inv(E[i])
        assert np.linalg.norm(got[i] - r) / np.linalg.norm(r) < 1e-13 * np.linalg.cond(E[i])
    assert not np.isfinite(got[1]).all() and not np.isfinite(got[3]).all()

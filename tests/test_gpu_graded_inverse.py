"""FP64 inverse of graded matrices.  Column scaling by powers of two is exact and changes
no pivot, so it must change no digit of the result; graded rows keep the bar of the
other FP64 inverse tests, 1e-13 x cond, column by column."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _inverse(E):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    with Chi0Plan(24, [g_sphere(E.shape[-1], (0.0, 0.0, 0.0))], np.zeros(len(E)), 1e-3, precision="fp64") as plan:
        t = plan.epsilon_inverse(0, torch.from_numpy(np.ascontiguousarray(E)).cuda()).cpu().numpy()
        plan.sync_status()
    return t


@pytest.mark.parametrize("n,span", [(40, 30), (64, 8), (130, 25), (257, 40), (300, 400)])
def test_column_scaling_changes_no_digit(n, span):
    rng = np.random.default_rng(n)
    A = np.eye(n) + 0.4 / np.sqrt(n) * (rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n)))
    A[2] = A[2] @ np.diag(np.logspace(0, -9, n)) @ A[1]         # beyond the refinement: the elimination's digits
    d = 2.0 ** rng.integers(-span, span + 1, n)
    got, base = _inverse(A * d), _inverse(A)
    assert np.array_equal(got * d[:, None], base)
    ref = np.linalg.inv(A[0])
    assert np.linalg.norm(base[0] - ref) / np.linalg.norm(ref) < 1e-13 * np.linalg.cond(A[0])


@pytest.mark.parametrize("n", [64, 200])
def test_graded_rows(n):
    rng = np.random.default_rng(n)
    A = np.eye(n) + 0.4 / np.sqrt(n) * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    d = 2.0 ** rng.integers(-6, 7, n)
    ref = np.linalg.inv(A)
    got = _inverse((d[:, None] * A)[None])[0] * d
    err = np.linalg.norm(got - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() < 1e-13 * np.linalg.cond(d[:, None] * A)

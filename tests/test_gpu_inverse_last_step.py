"""The refined FP64 inverse of matrices whose first residual is one large rank-one
term, I - (1 - e) / N 11^T (the rounding of its equal elements to FP32 points one
way): the error must be that of the FP64 elimination, which runs when the
refinement's memory is refused, up to the same rounding of the input, cond 2^-53."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,e", [(96, 2.0 ** -9), (300, 2.0 ** -12.3), (1000, 2.0 ** -14), (300, 2.0 ** -5.3),
                                 (1000, 2.0 ** -5.3)])
def test_coherent_residual(n, e, monkeypatch):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    c = (1.0 - e) / n
    diag = 1.0 - c
    # the matrix held is (diag + c) I - c 11^T: its inverse from exact rationals
    a, b = Fraction(diag) + Fraction(c), Fraction(c)
    ref = np.full((n, n), float(b / (a * (a - n * b))))
    ref[np.arange(n), np.arange(n)] += float(1 / a)
    E = np.full((1, n, n), -c, np.complex128)
    E[0, np.arange(n), np.arange(n)] = diag
    err = []
    for refuse in ("", "ws:%d" % (52 * n * n)):
        monkeypatch.setenv("CHI0_FAULT", refuse)
        with Chi0Plan(24, [g_sphere(n, (0.0, 0.0, 0.0))], [0.0], 1e-3, precision="fp64") as plan:
            got = plan.epsilon_inverse(0, torch.from_numpy(E.copy()).cuda())[0].cpu().numpy()
            plan.sync_status()
        err.append(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert err[0] <= max(2.0 * err[1], 2.0 ** -53 / float(a - n * b)), err

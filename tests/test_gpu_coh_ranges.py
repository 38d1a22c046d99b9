"""FP32 COH sums at the edges of their tiles and band chunks, with divisors inside
and outside the range of the bare reciprocal (poles 1e20 away, poles whose
imaginary part cancels delta).  Bar against the sum of the term magnitudes S as in
the other COH tests: 2e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nG,n_t,n_b,kind", [
    (1, 1, 1, "plain"), (32, 2, 32, "plain"), (33, 3, 33, "plain"), (65, 1, 97, "far"), (40, 2, 31, "cancel"),
])
def test_sigma_coh_ranges(nG, n_t, n_b, kind):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    rng = np.random.default_rng(nG)
    c = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    delta = 1e-3
    m = c(n_t * n_b, nG).astype(np.complex64)
    x, w, v = rng.standard_normal((n_t, n_b)), rng.uniform(0.5, 2, n_b), rng.uniform(0.1, 1, nG)
    Om, wt = c(nG, nG), rng.uniform(0.3, 3, (nG, nG)) + 0.3j * rng.standard_normal((nG, nG))
    if kind == "far":          # one pole far away, one without strength
        wt[3, 5], Om[7], wt[8, 9] = 1e20, 0.0, 0.0
    if kind == "cancel":       # x - wt + i delta is real for these
        wt[4] = wt[4].real + 1j * np.float64(np.float32(delta))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], [0.0], delta, precision="bf16") as plan:
        got = plan.sigma_coh(0, dev(m), n_t, n_b, dev(x), dev(Om), dev(wt), dev(v), w=dev(w))
    pole = (wt != 0) & (Om != 0)
    num = np.where(pole, Om * v[None] / (2 * np.where(pole, wt, 1)), 0)
    mm = m.astype(complex).reshape(n_t, n_b, nG)
    for t in range(n_t):
        terms = np.array([w[b] * mm[t, b][:, None] * num / (x[t, b] - wt + 1j * delta) * mm[t, b].conj()[None]
                          for b in range(n_b)])
        assert abs(got[t] - terms.sum()) <= 2e-6 * np.abs(terms).sum()

"""The dielectric inverse where its trailing update and look-ahead change form: odd
and even sizes around the 32-column panels and 64 x 64 tiles, several matrices,
rows that all move, and a call inside a CUDA graph capture (one stream) that gives
the same bits as the plain call.  Bars as in the other dielectric tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _plan(n_G, n_freq, precision):
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    return Chi0Plan(24, [g_sphere(n_G, (0.0, 0.0, 0.0))], np.zeros(n_freq), 1e-3, precision=precision)


@pytest.mark.parametrize("precision", ["bf16", "fp64"])
@pytest.mark.parametrize("n_G,n_freq", [(63, 1), (65, 3), (66, 1), (95, 2), (96, 2), (98, 1), (191, 1), (258, 5)])
def test_inverse_tile_edges(n_G, n_freq, precision):
    import torch
    rng = np.random.default_rng(n_G)
    E = rng.standard_normal((n_freq, n_G, n_G)) + 1j * rng.standard_normal((n_freq, n_G, n_G))
    E /= np.sqrt(n_G)
    for i in range(n_freq):        # large elements off the diagonal: every column interchanges rows
        E[i][rng.permutation(n_G), np.arange(n_G)] += 4.0
    ref = np.linalg.inv(E)
    with _plan(n_G, n_freq, precision) as plan:
        t = torch.from_numpy(E.copy()).cuda()
        plan.epsilon_inverse(0, t)
        plan.sync_status()
        got = t.cpu().numpy()
        graph, g2 = torch.cuda.CUDAGraph(), torch.from_numpy(E.copy()).cuda()
        work = g2.clone()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            work.copy_(g2)
            plan.epsilon_inverse(0, work)
        graph.replay()
        torch.cuda.synchronize()
        plan.sync_status()
        again = work.cpu().numpy()
    cond = max(np.linalg.cond(e) for e in E)
    tol = (1e-13 if precision == "fp64" else 2e-7 * np.sqrt(n_G)) * cond
    for i in range(n_freq):
        assert np.linalg.norm(got[i] - ref[i]) / np.linalg.norm(ref[i]) < tol
        assert np.linalg.norm(again[i] - ref[i]) / np.linalg.norm(ref[i]) < tol
    if precision != "fp64":
        assert np.array_equal(got, again)

"""The kernels that FP64 plans use where a workspace cannot be had: after a refused
allocation (CHI0_FAULT=ws:1) and inside a stream capture of a plan that has made no
call yet.  Both are the same route (equal bits), and no workspace grows.

References are FP64 products and NumPy FFTs.  The FP64 sums of at most 600 terms
carry some 10 x 2^-53 of their magnitudes, the direct transforms 6e-16: bar 1e-13."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _complex(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _rel(a, b):
    return np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)


def _both(make, call, monkeypatch):
    """call(plan) -> tensors: refused, then captured on a new plan; the refused call's result."""
    import torch
    monkeypatch.setenv("CHI0_FAULT", "ws:1")
    with make() as plan:
        held = plan.workspace_bytes
        ref = call(plan)
        plan.sync_status()
        assert plan.workspace_bytes == held
    monkeypatch.delenv("CHI0_FAULT")
    with make() as plan:
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            out = call(plan)
        graph.replay()
        torch.cuda.synchronize()
        assert plan.workspace_bytes == held
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
        plan.sync_status()
    return ref


@pytest.mark.parametrize("nG", [65, 300])
def test_contraction_and_dense_adjoint(nG, monkeypatch):
    from oracle import chi0_from_pairs, chi0_grad, freq_factor
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    rng = np.random.default_rng(nG)
    n_v, n_c, omega = 3, 200, np.array([0.0, 0.4j])
    M, Ev, Ec = _complex(rng, n_v * n_c, nG), -rng.uniform(0, 0.25, n_v), rng.uniform(0.2, 2.0, n_c)
    Gamma = _complex(rng, 2, nG, nG)
    dE = (Ev[:, None] - Ec[None]).reshape(-1)
    make = lambda: Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], omega, 1e-3, precision="fp64")
    args = [_dev(M), n_v, n_c, _dev(Ev), _dev(Ec)]
    chi, = _both(make, lambda p: [p.accumulate(0, *args)], monkeypatch)
    ref = chi0_from_pairs(M, freq_factor(dE, np.ones_like(dE), omega, 1e-3))
    for i in range(2):
        assert _rel(chi[i], ref[i]) < 1e-13
    Gd = _dev(Gamma)
    gM, gEv, gEc = _both(make, lambda p: p.backward(0, *args, grad_chi=Gd), monkeypatch)
    rM, rd = chi0_grad(M, dE, np.ones_like(dE), omega, 1e-3, Gamma)
    rd = rd.reshape(n_v, n_c)
    assert _rel(gM, rM) < 1e-13 and _rel(gEv, rd.sum(1)) < 1e-13 and _rel(gEc, -rd.sum(0)) < 1e-13


@pytest.mark.parametrize("n,half,n_v,n_c", [((24, 24, 24), 4, 2, 9), ((21, 27, 30), 5, 3, 4), ((96, 96, 96), 12, 1, 2),
                                            ((4, 120, 120), 1, 2, 3)])
def test_pairs(n, half, n_v, n_c, monkeypatch):
    """96^3 with 25 planes kept takes the FP64 kernel that goes through a plane in chunks of rows (188 KB as a whole); so
    does 120 x 120 always: it does not fit the fixed-point kernel either."""
    from paper_1601_06767_gb300 import Chi0Plan
    rng = np.random.default_rng(sum(n))
    ax = np.arange(-half, half + 1)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    g = g[(g ** 2).sum(1) <= half * half + 1]
    uv, uc = _complex(rng, n_v, *n), _complex(rng, n_c, *n)
    v, c = _dev(uv), _dev(uc)
    make = lambda: Chi0Plan(n, [g.astype(np.int32)], [0.0], 1e-3, precision="fp64")
    M, = _both(make, lambda p: [p.pairs(0, v, c)], monkeypatch)
    ref = np.array([np.fft.ifftn(a.conj() * b)[g[:, 0] % n[0], g[:, 1] % n[1], g[:, 2] % n[2]] for a in uv for b in uc])
    assert _rel(M, ref) < 1e-13

"""Workspaces made on demand: a captured inverse keeps its memory when a later call
outgrows it, a refusal (CHI0_FAULT=ws:N refuses N bytes and more) is not for
good, does not cost the workspace at hand and leaves capture possible."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _matrices(n, nf=1):
    rng = np.random.default_rng(n)
    return _dev(np.eye(n) + 0.3 / np.sqrt(n) * (rng.standard_normal((nf, n, n)) + 1j * rng.standard_normal((nf, n, n))))


def _plan(sizes, precision="fp64", n_freq=1):
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    return Chi0Plan(24, [g_sphere(n, (0.0, 0.0, 0.0)) for n in sizes], np.zeros(n_freq), 1e-3, precision=precision)


def _captured(plan, E):
    """A graph that inverts the matrices in the returned buffer in place."""
    import torch
    buf, graph = E.clone(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        plan.epsilon_inverse(0, buf)
    return graph, buf


@pytest.mark.parametrize("precision", ["fp64", "bf16"])
def test_captured_inverse_outlives_growth(precision):
    import torch
    small, large = _matrices(70), _matrices(300)
    with _plan([70, 300], precision) as plan:
        ref = plan.epsilon_inverse(0, small.clone())
        graph, buf = _captured(plan, small)
        held = plan.workspace_bytes
        big = plan.epsilon_inverse(1, large.clone())
        assert plan.workspace_bytes > held
        junk = torch.full((1 << 22,), 7, dtype=torch.int64, device="cuda")
        buf.copy_(small)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, ref) and int(junk.min()) == 7
        assert torch.equal(plan.epsilon_inverse(1, large.clone()), big)
        plan.sync_status()


def test_refused_refinement(monkeypatch):
    """128^2: the elimination needs 0.2 MB, the refinement 4 MB more."""
    import torch
    E = _matrices(128)
    bar = 1e-13 * float(torch.linalg.cond(E[0]))
    inv = torch.linalg.inv(E)
    rel = lambda a: float(torch.linalg.vector_norm(a - inv) / torch.linalg.vector_norm(inv))
    with _plan([128]) as plan:
        empty = plan.workspace_bytes
        monkeypatch.setenv("CHI0_FAULT", "ws:1000")
        with pytest.raises(Exception):
            plan.epsilon_inverse(0, E.clone())
        monkeypatch.setenv("CHI0_FAULT", "ws:1000000")
        first = plan.epsilon_inverse(0, E.clone())
        held = plan.workspace_bytes
        assert 0 < held - empty < 1000000
        graph, buf = _captured(plan, E)
        again = plan.epsilon_inverse(0, E.clone())
        assert plan.workspace_bytes == held and torch.equal(first, again)
        buf.copy_(E)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, first) and rel(first) < bar
        monkeypatch.delenv("CHI0_FAULT")
        assert rel(plan.epsilon_inverse(0, E.clone())) < bar
        assert plan.workspace_bytes > held + 1000000
        plan.sync_status()


def test_refused_contraction_is_asked_for_again(monkeypatch):
    import torch
    rng = np.random.default_rng(3)
    K, nG = 300, 150
    M = _dev(rng.integers(-99, 100, (K, nG)) + 1j * rng.integers(-99, 100, (K, nG)))
    Ev, Ec = _dev(np.zeros(1)), _dev(np.ones(K))
    ref = -(M.T @ M.conj())                                  # integers: exact on every route
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], [0.0], 0.0, precision="fp64") as plan:
        empty = plan.workspace_bytes
        monkeypatch.setenv("CHI0_FAULT", "ws:1000")
        assert torch.equal(plan.accumulate(0, M, 1, K, Ev, Ec)[0], ref) and plan.workspace_bytes == empty
        monkeypatch.delenv("CHI0_FAULT")
        assert torch.equal(plan.accumulate(0, M, 1, K, Ev, Ec)[0], ref) and plan.workspace_bytes > empty
        plan.sync_status()

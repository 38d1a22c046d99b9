"""Workspaces that FP64 plans allocate on demand: a captured call keeps its memory when a
later call outgrows it, and wavefunction transforms on several streams do not
overwrite each other's.  Equal calls give equal bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rand(rng, *shape):
    return _dev(rng.standard_normal(shape) + 1j * rng.standard_normal(shape))


def _g(lo, hi):
    ax = np.arange(lo, hi + 1)
    return np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)


def test_captured_pairs_outlive_growth():
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    rng = np.random.default_rng(1)
    n = (16, 18, 20)
    with Chi0Plan(n, [_g(-3, 3)], [0.0], 1e-3, precision="fp64") as plan:
        uv, uc = _rand(rng, 3, *n), _rand(rng, 9, *n)
        ref = plan.pairs(0, uv[:2], uc[:3])
        M = torch.zeros_like(ref)
        held = plan.workspace_bytes
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            plan.pairs(0, uv[:2], uc[:3], out=M)
        big = plan.pairs(0, uv, uc)
        assert plan.workspace_bytes > held
        junk = torch.full((1 << 24,), 7, dtype=torch.int64, device="cuda")
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(M, ref) and int(junk.min()) == 7
        assert torch.equal(plan.pairs(0, uv, uc), big)
        plan.sync_status()


def test_wavefunctions_on_several_streams():
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    rng = np.random.default_rng(2)
    g = _g(-6, 6)
    with Chi0Plan((24, 24, 24), [g[:1]], [0.0], 1e-3, precision="fp64", gw=g) as plan:
        coeff = [_rand(rng, 64, len(g)) for _ in range(3)]
        ref = [plan.wfn_to_grid(c) for c in coeff]
        streams = [torch.cuda.Stream() for _ in coeff]
        outs = [[torch.empty_like(r) for _ in range(6)] for r in ref]
        torch.cuda.synchronize()
        for k in range(6):
            for c, o, s in zip(coeff, outs, streams):
                with torch.cuda.stream(s):
                    plan.wfn_to_grid(c, out=o[k])
        graph, cap = torch.cuda.CUDAGraph(), torch.empty_like(ref[0])
        torch.cuda.synchronize()
        for r, o in zip(ref, outs):
            assert all(torch.equal(r, x) for x in o)
        with torch.cuda.graph(graph):          # direct sums inside a capture
            plan.wfn_to_grid(coeff[0], out=cap)
        graph.replay()
        torch.cuda.synchronize()
        plan.sync_status()
        # 13 + 13 + 13 terms summed in FP64 with rounded twiddles, and the fixed-point result's 2e-15
        assert float(torch.linalg.vector_norm(cap - ref[0]) / torch.linalg.vector_norm(ref[0])) < 1e-14

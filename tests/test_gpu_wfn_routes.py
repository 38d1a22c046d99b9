"""FP64 wavefunctions: a captured call gives the eager call's bits; bands of one large
and many small coefficients; subnormal numbers.

The error bar of a coefficient set: the columns' sums are rounded to 2^-56 of the
plane's largest, 2 x 13^2 of them, then two more transforms: sqrt(3 x 2 x 169) x
0.3 x 2^-55 = 5e-16 at most of the largest coefficient, whose modulus every |psi(r)| has here."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _plan(g, n=24):
    from paper_1601_06767_gb300 import Chi0Plan
    return Chi0Plan(n, [g[:1]], [0.0], 1e-3, precision="fp64", gw=g)


def _sphere():
    ax = np.arange(-6, 7)
    return np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)


def test_captured_bits():
    import torch
    g = _sphere()
    c = torch.randn((300, len(g)), dtype=torch.complex128, device="cuda")
    with _plan(g) as plan:
        ref = plan.wfn_to_grid(c)
        out, graph = torch.zeros_like(ref), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            plan.wfn_to_grid(c, out=out)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        plan.sync_status()


@pytest.mark.parametrize("small", [1e-2, 1e-4, 1e-9, 1e-20])
def test_one_large_coefficient(small):
    """Reference in extended precision: exact twiddles' products summed axis by axis."""
    import torch
    g, n = _sphere(), 24
    rng = np.random.default_rng(4)
    c = small * (rng.standard_normal(len(g)) + 1j * rng.standard_normal(len(g))) / np.sqrt(2 * len(g))
    c[777] = 0.6 - 0.8j
    with _plan(g) as plan:
        psi = plan.wfn_to_grid(torch.from_numpy(c[None]).cuda())[0].cpu().numpy()
    pi = np.longdouble("3.14159265358979323846264338327950288")
    w = np.exp(2j * pi * (np.arange(n)[:, None] * np.arange(-6, 7)[None] % n).astype(np.longdouble) / n)
    ref = c.reshape(13, 13, 13).astype(np.clongdouble)
    for axis in range(3):
        ref = np.moveaxis(np.tensordot(w, ref, (1, axis)), 0, axis)
    assert np.linalg.norm((psi - ref).astype(complex)) / np.linalg.norm(ref.astype(complex)) < 5e-16


def test_subnormal_coefficients():
    """Sums of subnormal numbers are exact where the twiddles are 1, -1, i, -i (a 2^3 grid)."""
    import torch
    ax = np.arange(0, 2)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    c = (np.arange(1, 9) - 3j) * 5e-324
    with _plan(g, 2) as plan:
        psi = plan.wfn_to_grid(torch.from_numpy(c[None]).cuda())[0].cpu().numpy()
    s = np.array([[1, 1], [1, -1]])
    ref = np.einsum("ax,by,cz,xyz->abc", s, s, s, np.arange(1, 9).reshape(2, 2, 2)), -3 * np.eye(1, 8).reshape(2, 2, 2) * 8
    assert np.array_equal(psi.real / 5e-324, ref[0]) and np.array_equal(psi.imag / 5e-324, ref[1])

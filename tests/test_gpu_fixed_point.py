"""Wavefunctions and pair elements of FP64 plans in fixed point, where the line transforms change
form: odd axes, even axes with odd and even halves, mixed grids, spheres away
from the origin (frequencies beyond n / 2, both ends of the range), pair blocks
in several chunks, and bands without a usable scale.

Reference: NumPy FFTs in FP64.  A plane's elements are rounded to 2^-56 of its
largest one three times; with a largest element of at most 30 times the rms that
is 3 x 30 x 2^-57 = 6e-16 of M, NumPy's own error included below 2e-15."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _plan(n, g, **kw):
    from paper_1601_06767_gb300 import Chi0Plan
    return Chi0Plan(n, [np.asarray(g, np.int32)], [0.0], 1e-3, precision="fp64", **kw)


def _ref(uv, uc, g, n):
    out = []
    for v in uv:
        for c in uc:
            f = np.fft.ifftn(v.conj() * c)
            out.append(f[g[:, 0] % n[0], g[:, 1] % n[1], g[:, 2] % n[2]])
    return np.array(out)


def _bands(rng, nb, n):
    return rng.standard_normal((nb,) + n) + 1j * rng.standard_normal((nb,) + n)


@pytest.mark.parametrize("n,lo,hi,max_pairs", [
    ((2, 2, 2), (0, 0, 0), (1, 1, 1), 0), ((3, 4, 5), (-1, -1, -2), (1, 2, 2), 0),
    ((6, 10, 22), (-3, -4, -5), (2, 5, 6), 0), ((8, 12, 24), (-4, -6, -12), (3, 5, 11), 0),
    ((24, 24, 24), (-4, -5, -4), (4, 4, 5), 64), ((21, 27, 30), (-3, 9, 11), (4, 15, 19), 0),
    ((48, 20, 33), (20, -3, -16), (27, 3, 16), 0), ((128, 4, 6), (-2, -2, -3), (3, 1, 2), 0),
    ((4, 7, 128), (-2, -3, -6), (1, 3, 6), 0), ((130, 4, 4), (-2, -1, -1), (2, 1, 1), 0),
])
def test_pairs_all_axis_forms(n, lo, hi, max_pairs):
    rng = np.random.default_rng(sum(n))
    g = np.stack(np.meshgrid(*[np.arange(a, b + 1) for a, b in zip(lo, hi)], indexing="ij"), -1).reshape(-1, 3)
    g = g[rng.permutation(len(g))[: max(1, (3 * len(g)) // 4)]]        # a sphere with holes, any order
    uv, uc = _bands(rng, 5, n), _bands(rng, 17, n)
    vi, ci = np.array([3, 0, 4, 1], np.int32), rng.permutation(17).astype(np.int32)
    ref = _ref(uv[vi], uc[ci], g, n)
    with _plan(n, g, max_pairs=max_pairs) as plan:
        M = plan.pairs(0, _dev(uv), _dev(uc), v_idx=_dev(vi), c_idx=_dev(ci)).cpu().numpy()
        plan.sync_status()
    assert np.linalg.norm(M - ref) / np.linalg.norm(ref) < 2e-15


def test_scales_zero_and_nonfinite_bands():
    """Bands many orders of magnitude apart, a band of zeros (exact zeros), and bands holding an infinity or
    a NaN: their pairs come out non-finite, the others are untouched.  A G vector listed twice is served too."""
    rng = np.random.default_rng(3)
    n, g = (12, 10, 9), np.array([[0, 0, 0], [1, -2, 3], [-1, 0, 2], [1, -2, 3]])
    uv, uc = _bands(rng, 4, n), _bands(rng, 5, n)
    uv *= np.array([1e-140, 1.0, 1e90, 1.0])[:, None, None, None]
    uc[1] = 0
    ref = _ref(uv, uc, g, n)
    for sphere in (g[:3], g):
        with _plan(n, sphere) as plan:
            M = plan.pairs(0, _dev(uv), _dev(uc)).cpu().numpy()
        r = ref[:, : len(sphere)]
        norm = np.linalg.norm(r, axis=1)
        assert np.all(np.linalg.norm(M - r, axis=1) <= 3e-15 * norm)
        assert not M.reshape(4, 5, -1)[:, 1].any()
    uv[1, 2, 3, 4], uc[3, 0, 0, 0] = np.inf, np.nan
    with _plan(n, g[:3]) as plan:
        fin = np.isfinite(plan.pairs(0, _dev(uv), _dev(uc)).cpu().numpy()).reshape(4, 5, -1)
    good = np.ones((4, 5), bool)
    good[1] = good[:, 3] = False
    assert np.all(fin[good]) and not fin[~good].any()


@pytest.mark.parametrize("n,lo,hi", [
    ((2, 2, 2), (0, 0, 0), (1, 1, 1)), ((3, 4, 5), (-1, -1, -2), (1, 2, 2)), ((6, 10, 22), (-2, -4, -10), (3, 5, 11)),
    ((24, 24, 24), (-7, -7, -7), (7, 7, 7)), ((21, 27, 30), (-6, 3, 11), (6, 11, 19)), ((48, 20, 33), (-14, -9, -16), (14, 6, 16)),
    ((130, 4, 4), (-3, -1, -1), (3, 1, 2)), ((70, 6, 4), (-34, -1, -1), (34, 1, 1)),
])
def test_wavefunctions_all_axis_forms(n, lo, hi):
    """psi(r) = sum_g c(g) exp(2 pi i g.r) against NumPy, bands far apart in magnitude, a zero band and one
    holding an infinity.  Three roundings to 2^-56 of a plane's largest value: bar 2e-15 as above."""
    rng = np.random.default_rng(sum(n) + 1)
    g = np.stack(np.meshgrid(*[np.arange(a, b + 1) for a, b in zip(lo, hi)], indexing="ij"), -1).reshape(-1, 3)
    g = g[rng.permutation(len(g))[: max(1, (2 * len(g)) // 3)]].astype(np.int32)
    c = rng.standard_normal((5, len(g))) + 1j * rng.standard_normal((5, len(g)))
    c *= np.array([1.0, 1e-120, 1e100, 0.0, 1.0])[:, None]
    ref = np.zeros((5,) + n, complex)
    for b in range(5):
        np.add.at(ref[b], tuple(np.mod(g, n).T), c[b])
        ref[b] = np.fft.ifftn(ref[b], norm="forward")
    c[4, 0] = np.inf
    from paper_1601_06767_gb300 import Chi0Plan
    with Chi0Plan(n, [np.zeros((1, 3), np.int32)], [0.0], 1e-3, precision="fp64", gw=g) as plan:
        psi = plan.wfn_to_grid(_dev(c)).cpu().numpy()
        plan.sync_status()
    for b in range(3):
        assert np.linalg.norm(psi[b] - ref[b]) <= 2e-15 * np.linalg.norm(ref[b])
    assert not psi[3].any() and not np.isfinite(psi[4]).any()

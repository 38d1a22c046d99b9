"""FP64 pair elements of bands localised apart: the largest product conj(psi_v) psi_c
is many orders below the product of the bands' peaks (slabs, molecules in a
cell, core-like states).  Each pair has its own accuracy.

Reference: NumPy FFTs in FP64.  A plane's or line's largest element is at most
sqrt(576) = 24 times its rms, so three roundings to 2^-56 of it are below 3 x 24 x 2^-57 = 5e-16
of M, and the products' two roundings on either side 2 x 2^-53: below 2e-15
together with NumPy's own sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _band(rng, n, centre, width):
    r2 = 0.0
    for a, c in zip(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), centre):
        d = (a - c + n / 2) % n - n / 2
        r2 = r2 + d * d
    return (rng.standard_normal((n, n, n)) + 1j * rng.standard_normal((n, n, n))) * np.exp(-r2 / (2 * width ** 2))


@pytest.mark.parametrize("shift,width", [
    ((8, 0, 0), 2.0), ((12, 0, 0), 1.6), ((0, 0, 12), 1.6), ((0, 12, 12), 1.6), ((12, 12, 12), 1.7), ((12, 12, 12), 1.4),
])
def test_bands_localised_apart(shift, width):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    rng = np.random.default_rng(int(10 * width) + sum(shift))
    n = 24
    ax = np.arange(-3, 4)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    v = np.stack([_band(rng, n, (5, 6, 7), width), _band(rng, n, (5, 6, 7), 50.0)])
    c = np.stack([_band(rng, n, np.add((5, 6, 7), shift), width), _band(rng, n, (0, 0, 0), 50.0)])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(n, [g], [0.0], 1e-3, precision="fp64") as plan:
        M = plan.pairs(0, dev(v), dev(c)).cpu().numpy().reshape(2, 2, -1)
        plan.sync_status()
    for i in range(2):
        for j in range(2):
            f = np.fft.ifftn(v[i].conj() * c[j])[g[:, 0], g[:, 1], g[:, 2]]
            assert np.linalg.norm(M[i, j] - f) < 2e-15 * np.linalg.norm(f), (i, j)

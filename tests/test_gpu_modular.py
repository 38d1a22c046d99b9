"""The FP64 contraction and the dense adjoint as modular products on the tensor
cores, at the edges of the tiles (256 x 256 outputs, 64-pair stages, 256-pair chains, pair blocks).

Integer pair elements and factors f = -w (omega = 0, delta = 0, dE = -1) make
every chi0 element an integer that FP64 matrix products give exactly.  The
kernels round nothing on such input; the reconstruction carries 2^-84 of the
moduli's product, at most 2^-80 of |M_G| |M_H|, and one rounding, so that is the
bar.  It also holds for the CUDA-core kernel, which small inputs keep."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _accumulate(M, w, n_freq=1, n=48, **kw):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    K, nG = M.shape
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(n, [g_sphere(nG, (0.0, 0.0, 0.0))], np.zeros(n_freq), 0.0, precision="fp64", **kw) as plan:
        chi = plan.accumulate(0, dev(M), 1, K, dev(np.zeros(1)), dev(np.ones(K)), dev(w))
        plan.sync_status()
        return chi.cpu().numpy()


@pytest.mark.parametrize("nG,K,n_freq,max_pairs,constant", [
    (1, 64, 1, 0, False), (31, 65, 2, 0, False), (33, 255, 1, 0, True), (128, 256, 1, 0, True),
    (255, 257, 1, 0, False), (256, 320, 2, 0, True), (257, 512, 3, 0, False), (513, 700, 1, 256, False),
    (300, 4096, 1, 0, True), (2200, 96, 2, 64, False),
])
def test_integer_sums_are_exact(nG, K, n_freq, max_pairs, constant):
    rng = np.random.default_rng(nG + K)
    M = rng.integers(-4000, 4001, (K, nG)) + 1j * rng.integers(-4000, 4001, (K, nG))
    if constant:      # rows of one value: every residue product of a chain has the same sign
        M = np.repeat(M[:1], K, 0)
    w = 2.0 ** rng.integers(0, 4, K)
    got = _accumulate(M, w, n_freq, max_pairs=max_pairs)
    ref = -((M.real * w[:, None]).T @ M.real + (M.imag * w[:, None]).T @ M.imag) \
        - 1j * ((M.imag * w[:, None]).T @ M.real - (M.real * w[:, None]).T @ M.imag)
    norm = np.sqrt((np.abs(M) ** 2).sum(0)) * 2.0 ** 3
    bar = 2.0 ** -52 * np.abs(ref) + 2.0 ** -80 * norm[:, None] * norm[None]
    for i in range(n_freq):
        assert np.all(np.abs(got[i].real - ref.real) <= bar) and np.all(np.abs(got[i].imag - ref.imag) <= bar)


def test_scales_zeros_and_nonfinite_rows():
    """Rows far apart in magnitude, a row of zeros (exact zeros result) and rows holding an infinity or a
    NaN (their rows and columns of chi0 come out non-finite, the rest stays exact)."""
    rng = np.random.default_rng(5)
    K, nG = 200, 70
    M = rng.integers(-4000, 4001, (K, nG)) + 1j * rng.integers(-4000, 4001, (K, nG))
    M[:, 5] = 0
    scale = 2.0 ** rng.integers(-400, 400, nG)
    Ms = M * scale
    ref = -(M.T @ M.conj())
    got = _accumulate(Ms, np.ones(K), n=24)[0] / scale[:, None] / scale[None]
    norm = np.sqrt((np.abs(M) ** 2).sum(0))
    assert np.all(np.abs(got - ref) <= 2.0 ** -51 * np.abs(ref) + 2.0 ** -79 * norm[:, None] * norm[None])
    assert not got[5].any() and not got[:, 5].any()
    Ms[3, 9], Ms[4, 11] = np.inf, np.nan
    bad = np.zeros(nG, bool)
    bad[[9, 11]] = True
    got = _accumulate(Ms, np.ones(K), n=24)[0]
    fin = np.isfinite(got.real) & np.isfinite(got.imag)
    assert np.all(fin[~bad][:, ~bad]) and not fin[bad].any() and not fin[:, bad].any()


@pytest.mark.parametrize("nG,n_v,n_c,n_freq,max_pairs,precision", [
    (63, 1, 1, 1, 0, "fp64"), (64, 3, 11, 2, 0, "fp64"), (129, 5, 51, 1, 0, "bf16"), (257, 7, 43, 3, 64, "fp64"),
    (300, 2, 128, 1, 0, "fp64"), (300, 9, 29, 2, 128, "fp16"),
])
def test_dense_adjoint_edges(nG, n_v, n_c, n_freq, max_pairs, precision):
    """Against FP64 matrix products.  Both sides carry a few sqrt(N_G) 2^-53 of the sums' magnitudes
    (5e-15 at N_G 300), so 1e-13; complex64 gradients one rounding of 2^-24 per frequency group."""
    import torch
    from oracle import chi0_grad
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    rng = np.random.default_rng(nG + n_v)
    K = n_v * n_c
    cdt = np.complex128 if precision == "fp64" else np.complex64
    M = (rng.standard_normal((K, nG)) + 1j * rng.standard_normal((K, nG))).astype(cdt)
    Ev, Ec, w = -rng.uniform(0, 0.25, n_v), rng.uniform(0.2, 2.0, n_c), rng.uniform(0.5, 2.0, n_c)
    omega = np.concatenate([[0.0], 1j * np.arange(1, n_freq)])
    Gamma = rng.standard_normal((n_freq, nG, nG)) + 1j * rng.standard_normal((n_freq, nG, nG))
    dE = (Ev[:, None] - Ec[None]).reshape(-1)
    rM, rd = chi0_grad(M.astype(complex), dE, np.tile(w, n_v), omega, 1e-3, Gamma)
    rd = rd.reshape(n_v, n_c)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with Chi0Plan(24, [g_sphere(nG, (0.0, 0.0, 0.0))], omega, 1e-3, precision=precision, max_pairs=max_pairs) as plan:
        gM, gEv, gEc = plan.backward(0, dev(M), n_v, n_c, dev(Ev), dev(Ec), dev(w), grad_chi=dev(Gamma))
        plan.sync_status()
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    assert rel(gM, rM) < (1e-13 if precision == "fp64" else 2.0 ** -24)
    assert rel(gEv, rd.sum(1)) < 1e-13 and rel(gEc, -rd.sum(0)) < 1e-13

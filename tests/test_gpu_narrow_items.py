"""Small contractions of split plans run as narrow items (128 x 64 or, with more
tiles, 128 x 128 of one component).  A plan with one frequency more than fit the chip that way
uses the next larger items (128 x 128 of one component, then of both): the same
sums in the same order, so the shared frequencies agree bit for bit off the diagonal
(whose FP64 sums are atomics).  The first frequency is compared with the FP64 sum."""
import numpy as np
import pytest

from oracle import chi0_from_pairs, freq_factor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("columns", [64, 128])
@pytest.mark.parametrize("precision,n_products,chain_pairs", [("bf16", 6, 0), ("bf16", 3, 96), ("fp16", 4, 0), ("fp16", 3, 64)])
@pytest.mark.parametrize("n_G,n_c", [(1, 1), (2, 40), (63, 33), (64, 7), (65, 160), (128, 32), (129, 301), (257, 64), (350, 96)])
def test_narrow_items_equal_full_tiles(n_G, n_c, precision, n_products, chain_pairs, columns):
    import torch
    from paper_1601_06767_gb300 import Chi0Plan
    from synth.mgo import g_sphere
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    fit = sms // (2 * ((n_G + 127) // 128) * ((n_G + columns - 1) // columns))
    assert fit >= 1
    rng = np.random.default_rng(n_G)
    g, n_v = g_sphere(n_G, (0.0, 0.0, 0.0)), 3
    omega = 0.3j * np.arange(1, fit + 2)
    M = rng.standard_normal((n_v * n_c, n_G)) + 1j * rng.standard_normal((n_v * n_c, n_G))
    E_v, E_c = np.sort(rng.uniform(-1.0, -0.1, n_v)), np.sort(rng.uniform(0.2, 3.0, n_c))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = []
    for om in (omega, omega[:fit]):
        with Chi0Plan((24, 24, 24), [g], om, 1e-3, precision=precision, n_products=n_products,
                      chain_pairs=chain_pairs, hermitian=False) as plan:
            chi = plan.new_chi(0)
            plan.accumulate(0, dev(M.astype(np.complex64)), n_v, n_c, dev(E_v), dev(E_c), chi=chi)
            plan.sync_status()
            out.append(chi.cpu().numpy())
    full, narrow = out[0][:fit], out[1]
    off = ~np.eye(n_G, dtype=bool)
    assert np.array_equal(full[:, off], narrow[:, off])
    d0, d1 = (np.einsum("wgg->wg", c) for c in (full, narrow))
    assert np.all(np.abs(d0 - d1) <= 1e-13 * np.abs(d0))
    # dropped products: 2^-16 of a product with two BF16 terms, 2^-22 with two FP16 terms; chains of up to
    # 96 pairs lose 1.4e-8 each per pair
    f = freq_factor((E_v[:, None] - E_c[None, :]).reshape(-1), np.ones(n_v * n_c), omega[:1], 1e-3)
    ref = chi0_from_pairs(M.astype(np.complex64).astype(complex), f)[0]
    tol = 4e-5 if (precision, n_products) == ("bf16", 3) else 4e-6
    assert np.linalg.norm(narrow[0] - ref) <= tol * np.linalg.norm(ref)

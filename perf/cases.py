"""The work that a user of this library has it do, as separately timed cases.

Every case goes through the public entry points of the package (Chi0Plan) on
inputs of the shapes and distributions of the library's own workloads: MgO-like
cells on a 24^3 (8-atom), 36^3, 48^3 (64-atom) or 96^3 (256-atom) grid, spheres
of 350 to 8000 G vectors, one static or up to 32 imaginary frequencies, FP64
plans (the default) and the split BF16 / FP16 plans.

listed()  the cases; draw(rng) one more of the same ranges; prepare / run one
pass; work what a pass cannot do without; exact the outputs in 64 bits.
"""
import math

import numpy as np
import torch

A0 = 7.96            # bohr, cubic cell at the 24^3 grid (scaled with the grid)
DELTA = 1e-3         # broadening, Hartree
E_LO, E_WIDTH = 0.17, 2.03   # conduction band edge and width, Hartree


def listed():
    return [
        # The 8-atom cell from coefficients to a static chi0 in split BF16: the smallest whole
        # calculation (a convergence scan runs many of them); launches and latency count.
        {"name": "path_8atom_bf16", "kind": "path", "precision": "bf16", "n": 24, "n_G": 350, "n_imag": 0,
         "n_v": 16, "n_c": 240, "max_pairs": 0, "weighted": False},
        # The same in the default precision: every reference calculation.
        {"name": "path_8atom_fp64", "kind": "path", "precision": "fp64", "n": 24, "n_G": 350, "n_imag": 0,
         "n_v": 16, "n_c": 240, "max_pairs": 0, "weighted": False},
        # One block of pair elements at the 64-atom size (valence set times 32 conduction bands).
        {"name": "pairs_64atom_split", "kind": "pairs", "precision": "bf16", "n": 48, "n_G": 2500,
         "n_v": 128, "n_c": 32},
        # Contraction of one 64-atom block, nine frequencies, columns of the accelerated sum (weights).
        {"name": "accumulate_64atom_bf16", "kind": "accumulate", "precision": "bf16", "n_G": 2500, "n_imag": 8,
         "n_v": 128, "n_c": 64, "weighted": True},
        # The same contraction in the default precision (a quarter of the pairs).
        {"name": "accumulate_64atom_fp64", "kind": "accumulate", "precision": "fp64", "n_G": 2500, "n_imag": 8,
         "n_v": 128, "n_c": 16, "weighted": False},
        # One block of the 256-atom calculation from coefficients: the largest workload, 16 selected
        # bands with weights, static and one imaginary frequency.
        {"name": "path_256atom_fp16", "kind": "path", "precision": "fp16", "n": 96, "n_G": 8000, "n_imag": 1,
         "n_v": 512, "n_c": 16, "max_pairs": 0, "weighted": True},
        # Eight shifted q-points with spheres of 2200 to 2600 vectors and 32 frequencies in one batched build.
        {"name": "batched_8q_fp16", "kind": "batched", "precision": "fp16", "n": 48, "n_q": 8, "n_G": 2200,
         "n_G_step": 57, "n_imag": 31, "n_v": 128, "n_c": 4},
        # Gradient of a loss on the diagonal of chi0 over all pairs of the 36^3 workload.
        {"name": "adjoint_diag_fp16", "kind": "adjoint_diag", "precision": "fp16", "n_G": 1200, "n_imag": 0,
         "n_v": 64, "n_c": 2000},
        # Gradient of a loss on the whole matrix (what autograd through the contraction calls).
        {"name": "adjoint_dense_fp64", "kind": "adjoint_dense", "precision": "fp64", "n_G": 1200, "n_imag": 0,
         "n_v": 64, "n_c": 64},
        # Dielectric matrices of the 64-atom sphere and their inverses, nine frequencies, split plan.
        {"name": "inverse_64atom_split", "kind": "inverse", "precision": "bf16", "n_G": 2500, "n_imag": 8},
        # Static dielectric matrix and inverse in the default precision.
        {"name": "inverse_static_fp64", "kind": "inverse", "precision": "fp64", "n_G": 1200, "n_imag": 0},
        # Coulomb-hole self-energy of four bands with the accelerated band sum at the 64-atom size.
        {"name": "coh_64atom_split", "kind": "coh", "precision": "bf16", "n_G": 2500, "n_t": 4, "n_b": 663},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "pairs", "accumulate", "accumulate", "batched", "adjoint_diag", "adjoint_dense",
                       "inverse", "coh"])
    precision = rng.choice(["fp64", "bf16", "fp16"])
    wide = precision == "fp64"
    c = {"kind": kind, "precision": precision}
    if kind in ("path", "pairs"):
        # even, odd and ragged grids; the largest only with few pairs in 64 bits
        n = rng.choice([21, 24, 24, 30, 36, 45, 48, 48, 96])
        top = {21: 300, 24: 400, 30: 700, 36: 1200, 45: 2200, 48: 2600, 96: 8000}[n]
        c.update(n=n, n_G=_log_int(rng, max(57, top // 8), top), n_v=_log_int(rng, 1, 256 if n == 96 else 128))
        most = {21: 8192, 24: 8192, 30: 8192, 36: 4096, 45: 2048, 48: 4096, 96: 1024}[n]
        if wide:
            most = min(most, 200 if n == 96 else 2048)
        c["n_v"] = min(c["n_v"], most)
        c["n_c"] = _log_int(rng, 1, max(1, most // c["n_v"]))
        if kind == "path":
            c.update(n_imag=rng.choice([0, 0, 1, 2, 8]), weighted=rng.random() < 0.5,
                     max_pairs=rng.choice([0, 0, 0, 1024]))
            if wide and n > 48:
                c["n_imag"] = 0
    elif kind == "accumulate":
        c.update(n_G=_log_int(rng, 100, 3000), n_imag=rng.choice([0, 1, 2, 4, 8, 15]), n_v=_log_int(rng, 1, 512),
                 weighted=rng.random() < 0.5)
        c["n_c"] = _log_int(rng, 1, max(1, 8192 // c["n_v"]))
        flops = 8.0 * c["n_G"] ** 2 * (1 + c["n_imag"]) * c["n_v"]
        c["n_c"] = max(1, min(c["n_c"], int((4e11 if wide else 4e12) / flops)))
    elif kind == "batched":
        c.update(n=rng.choice([24, 36, 48]), n_q=rng.randint(2, 8), n_imag=rng.choice([0, 1, 7, 15, 31]),
                 n_v=_log_int(rng, 4, 128))
        top = {24: 350, 36: 1200, 48: 2200}[c["n"]]
        c["n_G"] = _log_int(rng, 100, top)
        c["n_G_step"] = rng.randint(0, max(1, c["n_G"] // 32))
        c["n_c"] = rng.randint(1, 8)
        if wide:
            c["n_imag"] = min(c["n_imag"], 1)
            c["n_v"] = min(c["n_v"], 16)
    elif kind == "adjoint_diag":
        c.update(n_G=_log_int(rng, 100, 2500), n_imag=rng.choice([0, 0, 1, 8]), n_v=_log_int(rng, 1, 128))
        c["n_c"] = _log_int(rng, 1, max(1, int(6e7 / c["n_G"] / c["n_v"])))
    elif kind == "adjoint_dense":
        c.update(n_G=_log_int(rng, 100, 2500), n_imag=rng.choice([0, 0, 1, 8]), n_v=_log_int(rng, 1, 64))
        c["n_c"] = max(1, min(_log_int(rng, 1, 128),
                              int(2e11 / (16.0 * c["n_G"] ** 2 * (1 + c["n_imag"]) * c["n_v"]))))
    elif kind == "inverse":
        c.update(n_G=_log_int(rng, 100, 1500 if wide else 2500), n_imag=rng.choice([0, 1, 2, 8]))
    else:
        c.update(n_G=_log_int(rng, 100, 1200 if wide else 2500), n_t=rng.randint(1, 8),
                 n_b=_log_int(rng, 10, 60 if wide else 700))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sphere(n_G, q=(0.0, 0.0, 0.0)):
    """The n_G integer vectors with the smallest |q + g|^2."""
    r = int(math.ceil((3.0 * n_G / (4.0 * math.pi)) ** (1.0 / 3.0))) + 3
    ax = np.arange(-r, r + 1)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    k2 = np.round(((g + np.asarray(q)[None, :]) ** 2).sum(1), 9)
    order = np.lexsort((g[:, 2], g[:, 1], g[:, 0], k2))
    return np.ascontiguousarray(g[order[:n_G]].astype(np.int32))


def _wfn_sphere(n):
    r = int(7 * n / 24)
    ax = np.arange(-r, r + 1)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    return np.ascontiguousarray(g[(g * g).sum(1) <= (7.0 * n / 24.0) ** 2 + 1e-9].astype(np.int32))


def _q_points(n_q):
    """Points of the shifted 2 x 2 x 2 grid."""
    return [((i // 4 + 0.5) / 2, (i // 2 % 2 + 0.5) / 2, (i % 2 + 0.5) / 2) for i in range(n_q)]


def _omega(n_imag):
    if n_imag == 0:
        return np.zeros(1, np.complex128)
    return np.concatenate([[0.0], 1j * np.logspace(-2, math.log10(2.0), n_imag)])


def _small_grid(n_G):
    """A grid that holds the sphere, for plans that only contract."""
    for n in (24, 36, 48, 96):
        if 2 * (3.0 * n_G / (4.0 * math.pi)) ** (1.0 / 3.0) + 4 < n:
            return n
    return 96


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(gen, shape, dtype=torch.complex128):
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device="cuda", dtype=real))


def _uniform(gen, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)


def _coeff(gen, nb, npw):
    """Normalised complex Gaussian plane-wave coefficients."""
    c = _normal(gen, (nb, npw))
    return c / torch.linalg.vector_norm(c, dim=1, keepdim=True)


def _grids(coeff, gw, n):
    """psi(r) = sum_g c(g) exp(2 pi i g.r) in 64 bits."""
    idx = torch.from_numpy(np.mod(gw.astype(np.int64), n)).cuda()
    flat = (idx[:, 0] * n + idx[:, 1]) * n + idx[:, 2]
    out = torch.empty((coeff.shape[0], n, n, n), dtype=torch.complex128, device="cuda")
    step = max(1, int(2e8 / n ** 3))
    for b in range(0, coeff.shape[0], step):
        box = torch.zeros((min(step, coeff.shape[0] - b), n ** 3), dtype=torch.complex128, device="cuda")
        box[:, flat] = coeff[b:b + step]
        out[b:b + step] = torch.fft.ifftn(box.view(-1, n, n, n), dim=(1, 2, 3), norm="forward")
    return out


def _energies(gen, n_v, n_c):
    """Valence energies over a 0.25 Ha band, conduction energies a run of neighbouring bands of a
    square-root density of states, both slightly scattered."""
    j = torch.arange(n_v, device="cuda", dtype=torch.float64)
    E_v = -0.25 + 0.25 * (j + _uniform(gen, (n_v,), 0.25, 0.75)) / n_v
    x0 = _uniform(gen, (1,), 0.02, 0.9)
    j = torch.arange(n_c, device="cuda", dtype=torch.float64)
    x = (x0 + 0.1 * (j + _uniform(gen, (n_c,), 0.25, 0.75)) / n_c).clamp(max=1.0)
    return E_v, (E_LO + E_WIDTH * x ** (2.0 / 3.0)).contiguous()


def _pair_matrix(gen, n_p, g, dtype):
    """Gaussian pair elements under an envelope falling with |G|."""
    env = 0.02 / (1.0 + torch.from_numpy((g.astype(np.float64) ** 2).sum(1)).cuda() / 16.0)
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    return _normal(gen, (n_p, g.shape[0]), dtype) * env.to(real)[None]


def _make(case, seed):
    """The inputs of a case (tensors on the GPU), the same for prepare and exact."""
    gen, kind = _gen(seed), case["kind"]
    wide = case["precision"] == "fp64"
    cdtype = torch.complex128 if wide else torch.complex64
    d = {"omega": _omega(case.get("n_imag", 0))}
    if kind in ("path", "pairs", "batched"):
        n = case["n"]
        d["n"], d["gw"] = n, _wfn_sphere(n)
        npw = d["gw"].shape[0]
        n_v, n_c = case["n_v"], case["n_c"]
        if kind == "batched":
            d["g"] = [_sphere(case["n_G"] + case["n_G_step"] * i, q) for i, q in enumerate(_q_points(case["n_q"]))]
            d["psi_c"] = _grids(_coeff(gen, n_c, npw), d["gw"], n).to(cdtype)
            d["psi_v"] = [_grids(_coeff(gen, n_v, npw), d["gw"], n).to(cdtype) for _ in d["g"]]
            d["E_v"], d["E_c"] = [], None
            for _ in d["g"]:
                E_v, E_c = _energies(gen, n_v, n_c)
                d["E_v"].append(E_v)
            d["E_c"] = E_c
            return d
        d["g"] = [_sphere(case["n_G"])]
        if kind == "pairs":
            d["psi_v"] = _grids(_coeff(gen, n_v, npw), d["gw"], n).to(cdtype)
            d["psi_c"] = _grids(_coeff(gen, n_c, npw), d["gw"], n).to(cdtype)
            return d
        d["c_v"], d["c_c"] = _coeff(gen, n_v, npw), _coeff(gen, n_c, npw)
        d["E_v"], d["E_c"] = _energies(gen, n_v, n_c)
        d["w"] = _uniform(gen, (n_c,), 0.5, 20.0) if case["weighted"] else None
        # a selection names its bands: columns in another order than the grids
        d["c_idx"] = torch.randperm(n_c, generator=gen, device="cuda").to(torch.int32) if case["weighted"] else None
        return d
    d["g"] = [_sphere(case["n_G"])]
    d["n"] = _small_grid(case["n_G"])
    n_G, nf = case["n_G"], d["omega"].size
    if kind in ("accumulate", "adjoint_diag", "adjoint_dense"):
        n_v, n_c = case["n_v"], case["n_c"]
        d["M"] = _pair_matrix(gen, n_v * n_c, d["g"][0], cdtype)
        d["E_v"], d["E_c"] = _energies(gen, n_v, n_c)
        d["w"] = _uniform(gen, (n_c,), 0.5, 20.0) if case.get("weighted") else None
        if kind == "adjoint_diag":
            d["diag"] = _uniform(gen, (nf, n_G), 0.0, 1.0)
        if kind == "adjoint_dense":
            d["gamma"] = _normal(gen, (nf, n_G, n_G))
    elif kind == "inverse":
        # negative semidefinite static chi0, damped along the imaginary axis, and v = 4 pi / (Omega |q+G|^2)
        X = _normal(gen, (n_G // 2 + 1, n_G), torch.complex64) / math.sqrt(n_G)
        f = (_uniform(gen, (n_G // 2 + 1,), 0.2, 1.0)).to(torch.float32)
        d["chi"] = torch.empty((nf, n_G, n_G), dtype=torch.complex128, device="cuda")
        for i, om in enumerate(d["omega"]):
            fw = -f / (1.0 + abs(om) ** 2 / f)
            d["chi"][i] = (X.T * torch.complex(fw, DELTA * fw)[None]) @ X.conj()
        k2 = torch.from_numpy(((d["g"][0] + np.array([0.05, 0.0, 0.0])) ** 2).sum(1)).cuda()
        d["v"] = (4.0 / k2).contiguous()
    else:
        n_t, n_b = case["n_t"], case["n_b"]
        d["m"] = _pair_matrix(gen, n_t * n_b, d["g"][0], cdtype)
        E_t = _uniform(gen, (n_t,), 0.2, 0.6)
        d["x"] = (E_t[:, None] - _uniform(gen, (n_b,), -0.25, 2.2).sort().values[None]).contiguous()
        d["w"] = _uniform(gen, (n_b,), 0.5, 20.0)
        d["Om2"] = 0.3 * _normal(gen, (n_G, n_G))
        d["wt"] = torch.complex(_uniform(gen, (n_G, n_G), 0.3, 3.0), _uniform(gen, (n_G, n_G), -0.4, 0.4))
        k2 = torch.from_numpy(((d["g"][0] + np.array([0.05, 0.0, 0.0])) ** 2).sum(1)).cuda()
        d["v"] = (4.0 / k2).contiguous()
    return d


# ---------------------------------------------------------------------------
# one pass through the library
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_1601_06767_gb300 import Chi0Plan
    d = _make(case, seed)
    d["case"] = case
    d["plan"] = Chi0Plan(d["n"], d["g"], d["omega"], DELTA, precision=case["precision"], gw=d.get("gw"),
                         max_pairs=case.get("max_pairs", 0))
    if case["kind"] == "batched":   # kept by the caller between builds, as the captured graph expects
        d["chis"] = [d["plan"].new_chi(i) for i in range(case["n_q"])]
    return d


def run(state):
    s, plan, case = state, state["plan"], state["case"]
    kind = case["kind"]
    if kind == "pairs":
        return plan.pairs(0, s["psi_v"], s["psi_c"])
    if kind == "path":
        psi_v, psi_c = plan.wfn_to_grid(s["c_v"]), plan.wfn_to_grid(s["c_c"])
        return plan.build(0, psi_v, s["E_v"], psi_c, s["E_c"], w_col=s["w"], c_idx=s["c_idx"])
    if kind == "accumulate":
        return plan.accumulate(0, s["M"], case["n_v"], case["n_c"], s["E_v"], s["E_c"], s["w"])
    if kind == "batched":
        for c in s["chis"]:
            c.zero_()
        return plan.build_batched(s["psi_v"], s["E_v"], s["psi_c"], s["E_c"], chis=s["chis"])
    if kind == "adjoint_diag":
        return plan.backward(0, s["M"], case["n_v"], case["n_c"], s["E_v"], s["E_c"], diag_g=s["diag"])
    if kind == "adjoint_dense":
        return plan.backward(0, s["M"], case["n_v"], case["n_c"], s["E_v"], s["E_c"], grad_chi=s["gamma"])
    if kind == "inverse":
        return plan.epsilon_inverse(0, plan.epsilon(0, s["chi"], s["v"], symmetric=True))
    return plan.sigma_coh(0, s["m"], case["n_t"], case["n_b"], s["x"], s["Om2"], s["wt"], s["v"], w=s["w"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind, cb = case["kind"], 16 if case["precision"] == "fp64" else 8
    nf, n_G = 1 + case.get("n_imag", 0), case["n_G"]
    if kind in ("path", "pairs", "batched"):
        nr = case["n"] ** 3
        npw = 4.0 / 3.0 * math.pi * (7.0 * case["n"] / 24.0) ** 3
        n_p = case["n_v"] * case["n_c"]
        fft = 5.0 * nr * math.log2(nr)
        if kind == "pairs":
            return {"bytes": float((case["n_v"] + case["n_c"]) * nr * cb + n_p * n_G * cb),
                    "flops": n_p * (6.0 * nr + fft)}
        if kind == "path":
            nb = case["n_v"] + case["n_c"]
            return {"bytes": nb * npw * 16 + nf * n_G ** 2 * 16.0,
                    "flops": nb * fft + n_p * (6.0 * nr + fft) + 8.0 * n_G ** 2 * n_p * nf}
        gs = [n_G + case["n_G_step"] * i for i in range(case["n_q"])]
        return {"bytes": (case["n_q"] * case["n_v"] + case["n_c"]) * nr * cb + sum(nf * g ** 2 * 16.0 for g in gs),
                "flops": sum(n_p * (6.0 * nr + fft) + 8.0 * g ** 2 * n_p * nf for g in gs)}
    if kind == "inverse":
        return {"bytes": 2.0 * 16 * nf * n_G ** 2, "flops": 8.0 * n_G ** 3 * nf}
    if kind == "coh":
        n_p = case["n_t"] * case["n_b"]
        return {"bytes": n_p * n_G * cb + 2.0 * 16 * n_G ** 2, "flops": 22.0 * n_p * n_G ** 2}
    n_p = case["n_v"] * case["n_c"]
    if kind == "accumulate":
        return {"bytes": n_p * n_G * cb + nf * n_G ** 2 * 16.0, "flops": 8.0 * n_G ** 2 * n_p * nf}
    if kind == "adjoint_diag":
        return {"bytes": 2.0 * n_p * n_G * cb, "flops": n_p * n_G * (2.0 + 6.0 * nf)}
    return {"bytes": 2.0 * n_p * n_G * cb + nf * n_G ** 2 * 16.0, "flops": 16.0 * n_G ** 2 * n_p * nf}


# ---------------------------------------------------------------------------
# the outputs in 64 bits, with plain torch
# ---------------------------------------------------------------------------
def _factors(E_v, E_c, w, omega, n_v, n_c, derivative=False):
    dE = (E_v[:, None] - E_c[None, :]).reshape(-1).to(torch.complex128)
    wp = torch.ones(n_c, dtype=torch.float64, device="cuda") if w is None else w
    wp = wp[None].expand(n_v, n_c).reshape(-1)
    out = []
    for om in omega:
        a, b = dE - complex(om) + 1j * DELTA, dE + complex(om) + 1j * DELTA
        out.append(-0.5 * wp * (a ** -2 + b ** -2) if derivative else 0.5 * wp * (1 / a + 1 / b))
    return out


def _pair_elements(psi_v, psi_c, g, n):
    idx = torch.from_numpy(np.mod(g.astype(np.int64), n)).cuda()
    flat = (idx[:, 0] * n + idx[:, 1]) * n + idx[:, 2]
    n_v, n_c = psi_v.shape[0], psi_c.shape[0]
    M = torch.empty((n_v, n_c, g.shape[0]), dtype=torch.complex128, device="cuda")
    step = max(1, int(3e8 / n ** 3))
    for v in range(n_v):
        for c in range(0, n_c, step):
            x = psi_v[v].to(torch.complex128).conj()[None] * psi_c[c:c + step].to(torch.complex128)
            M[v, c:c + step] = torch.fft.ifftn(x, dim=(1, 2, 3)).reshape(x.shape[0], -1)[:, flat]
    return M.reshape(n_v * n_c, -1)


def _contract(M, fs):
    chi = torch.zeros((len(fs), M.shape[1], M.shape[1]), dtype=torch.complex128, device="cuda")
    for p in range(0, M.shape[0], 1024):
        B = M[p:p + 1024].to(torch.complex128)
        for i, f in enumerate(fs):
            chi[i].addmm_((B * f[p:p + 1024, None]).T, B.conj())
    return chi


def exact(case, seed):
    if case["kind"] in ("path", "accumulate", "batched") and work(case)["flops"] > 1.2e13:
        return None
    d = _make(case, seed)
    kind, n_v, n_c = case["kind"], case.get("n_v"), case.get("n_c")
    if kind == "pairs":
        return _pair_elements(d["psi_v"], d["psi_c"], d["g"][0], d["n"])
    if kind == "path":
        psi_v, psi_c = _grids(d["c_v"], d["gw"], d["n"]), _grids(d["c_c"], d["gw"], d["n"])
        if d["c_idx"] is not None:
            psi_c = psi_c[d["c_idx"].long()]
        M = _pair_elements(psi_v, psi_c, d["g"][0], d["n"])
        return _contract(M, _factors(d["E_v"], d["E_c"], d["w"], d["omega"], n_v, n_c))
    if kind == "batched":
        return [_contract(_pair_elements(p, d["psi_c"], g, d["n"]),
                          _factors(e, d["E_c"], None, d["omega"], n_v, n_c))
                for p, e, g in zip(d["psi_v"], d["E_v"], d["g"])]
    if kind == "accumulate":
        return _contract(d["M"], _factors(d["E_v"], d["E_c"], d["w"], d["omega"], n_v, n_c))
    if kind in ("adjoint_diag", "adjoint_dense"):
        fs = _factors(d["E_v"], d["E_c"], d["w"], d["omega"], n_v, n_c)
        fd = _factors(d["E_v"], d["E_c"], d["w"], d["omega"], n_v, n_c, derivative=True)
        gM = torch.empty_like(d["M"], dtype=torch.complex128)
        gd = torch.empty(n_v * n_c, dtype=torch.float64, device="cuda")
        for p in range(0, n_v * n_c, 16384):
            M = d["M"][p:p + 16384].to(torch.complex128)
            out, dE = torch.zeros_like(M), 0.0
            for i in range(len(fs)):
                f, df = fs[i][p:p + 16384, None], fd[i][p:p + 16384]
                if kind == "adjoint_diag":
                    GM = d["diag"][i][None] * M
                    out += 2.0 * f.real * GM
                else:
                    GM = M @ d["gamma"][i].T
                    out += f.conj() * GM + f * (M @ d["gamma"][i].conj())
                dE = dE + (df * (M.conj() * GM).sum(1).conj()).real
            gM[p:p + 16384], gd[p:p + 16384] = out, dE
        gd = gd.reshape(n_v, n_c)
        return gM, gd.sum(1), -gd.sum(0)
    if kind == "inverse":
        s = d["v"].sqrt()
        eye = torch.eye(case["n_G"], dtype=torch.complex128, device="cuda")
        return torch.stack([torch.linalg.inv(eye - s[:, None] * c * s[None]) for c in d["chi"]])
    sigma = torch.zeros(case["n_t"], dtype=torch.complex128, device="cuda")
    num = d["Om2"] * d["v"][None] / (2.0 * d["wt"])
    m = d["m"].to(torch.complex128).reshape(case["n_t"], case["n_b"], -1)
    for t in range(case["n_t"]):
        for b in range(case["n_b"]):
            K = num / (d["x"][t, b] - d["wt"] + 1j * DELTA)
            sigma[t] += d["w"][b] * (m[t, b] @ (K @ m[t, b].conj()))
    return sigma.cpu().numpy()

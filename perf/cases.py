"""The work a user of this framework has it do, as measurable cases.

Every case is one call of a public entry point (the binding of include/dmet_emb.h) on device-resident inputs, with the
plan made beforehand as a program that calls it in a loop keeps it. Kinds:

  eri          dmet_emb_eri of one problem: FP64 (the default precision) and the tensor-core precisions, real orbitals
               (8-fold packed) and complex ones (dense), restricted and unrestricted, full and reduced L
  batch        dmet_emb_eri of a plan of many uneven problems, replayed from a CUDA graph
  three_index  dmet_emb_transform_3idx: the embedded factors of a solver that takes density-fitted integrals
  jk           dmet_emb_jk_df: Coulomb and exchange straight from those factors
  fock, bath   dmet_emb_fock and dmet_emb_bath: the one-particle Hamiltonian and the embedding orbitals
  fftdf        dmet_emb_eri_fftdf: the plane-wave variant

Inputs are drawn on the GPU from the seed: real-space-real integrals that decay with the cell distance and are
Fourier-transformed to the k mesh, orthonormal orbitals, idempotent density matrices, Gaussian AOs on a grid.
"""
import math

import numpy as np
import torch

import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

C128, F64 = torch.complex128, torch.float64
PREC = {"fp64": B.DMET_PREC_FP64, "bf16x3": B.DMET_PREC_BF16X3, "tf32": B.DMET_PREC_TF32,
        "tf32x3": B.DMET_PREC_TF32X3, "fp16x2": B.DMET_PREC_FP16X2}


def _eri(name, mesh, n_ao, n_aux, n_emb, prec, n_emb_b=0, orbitals="real", reduced=False, decay=0.6, log_range=0.0):
    c = {"kind": "eri", "mesh": "x".join(map(str, mesh)), "n_ao": n_ao, "n_aux": n_aux, "n_emb": n_emb,
         "n_emb_b": n_emb_b, "prec": prec, "orbitals": orbitals, "reduced": reduced, "decay": decay,
         "log_range": log_range}
    return dict(c, name=name) if name else c


def listed():
    hbn = {"mesh": "6x6x1", "n_ao": 26, "n_aux": 220, "n_emb": 104}
    return [
        # the smallest complete problem (a model cell on 2x2x1): launches and latency count
        _eri("eri_fp64_tiny", (2, 2, 1), 8, 40, 16, "fp64", decay=0.7),
        # the embedding orbitals from the mean-field density, once per self-consistency step (h-BN-shaped)
        {"name": "bath_hbn", "kind": "bath", "mesh": "6x6x1", "n_ao": 26, "n_val": 24},
        # the embedding Fock matrix from the packed ERI, once per self-consistency step (h-BN-shaped)
        {"name": "fock_hbn", "kind": "fock", "mesh": "6x6x1", "n_ao": 26, "n_emb": 104},
        # one embedding problem in the default precision, FP64 (h-BN-shaped)
        _eri("eri_fp64_hbn", (6, 6, 1), 26, 220, 104, "fp64", decay=0.5),
        # the same problem on the tensor-core precision that production runs use
        _eri("eri_bf16x3_hbn", (6, 6, 1), 26, 220, 104, "bf16x3", decay=0.5),
        # a large restricted problem with reduced L and a wide range of orbital coefficients (silicon-shaped)
        _eri("eri_bf16x3_si", (4, 4, 4), 52, 400, 200, "bf16x3", reduced=True, log_range=4.0),
        # an unrestricted problem (aa, ab and bb blocks) of odd sizes on the fastest split (a transition-metal oxide)
        _eri("eri_fp16x2_uhf", (4, 4, 1), 52, 417, 119, "fp16x2", n_emb_b=113),
        # complex orbitals (no time-reversal symmetry): the dense complex ERI
        _eri("eri_bf16x3_complex", (6, 6, 1), 26, 220, 104, "bf16x3", orbitals="complex", decay=0.5),
        # many small uneven problems at once (a scan over fragments or geometries), replayed from a graph
        {"name": "batch24_bf16x3", "kind": "batch", "n_problems": 24, "shapes": 4000, "n_ao_min": 6, "n_ao_max": 12,
         "n_emb_min": 16, "n_emb_max": 48, "prec": "bf16x3"},
        # the embedded factors for a density-fitting solver, odd sizes, FP64
        {"name": "three_index_fp64", "kind": "three_index", "mesh": "3x3x2", "n_ao": 17, "n_aux": 145, "n_emb": 61,
         "prec": "fp64"},
        # Coulomb and exchange of one density from those factors, every solver iteration (h-BN-shaped)
        dict({k: hbn[k] for k in ("mesh", "n_aux", "n_emb")}, name="jk_df_hbn", kind="jk"),
        # the plane-wave variant on a small cell
        {"name": "fftdf_2x2x2", "kind": "fftdf", "mesh": "2x2x2", "n_ao": 8, "grid": 12, "n_emb": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind, then sizes spread over the logarithm of their ranges, kept below the listed cases' cost."""
    kind = rng.choice(["fp64", "fp64", "tensor", "tensor", "tensor", "complex", "three_index", "jk", "fock", "bath",
                       "fftdf", "batch"])
    while True:
        mesh = rng.choice([(1, 1, 1), (2, 1, 1), (2, 2, 1), (3, 2, 1), (2, 2, 2), (3, 3, 1), (3, 3, 2), (4, 4, 1),
                           (5, 3, 1), (3, 3, 3), (6, 6, 1), (4, 4, 3)])
        nk, ms = math.prod(mesh), "x".join(map(str, mesh))
        n_ao = _log(rng, 4, 60)
        n_aux = int(n_ao * rng.uniform(5.0, 10.0))
        n = min(_log(rng, 8, 160), nk * n_ao)
        decay = round(rng.uniform(0.4, 0.8), 3)
        if kind in ("fp64", "tensor", "complex"):
            prec = "fp64" if kind == "fp64" else rng.choice(["bf16x3", "bf16x3", "bf16x3", "fp16x2", "tf32x3", "tf32"])
            uhf = kind != "complex" and rng.random() < 0.4
            nb = max(1, min(nk * n_ao, n - rng.randint(0, 7))) if uhf else 0
            c = _eri(None, mesh, n_ao, n_aux, n, prec, nb, "complex" if kind == "complex" else "real",
                     kind != "complex" and rng.random() < 0.3, decay, rng.choice([0.0, 0.0, 2.0]))
            cap = 0.2e12 if kind == "fp64" else 3e12
        elif kind == "three_index":
            c = {"kind": kind, "mesh": ms, "n_ao": n_ao, "n_aux": n_aux, "n_emb": n,
                 "prec": rng.choice(["fp64", "fp64", "bf16x3"])}
            cap = 0.2e12
        elif kind == "jk":
            c = {"kind": kind, "mesh": ms, "n_aux": n_aux, "n_emb": n}
            cap = 0.15e12
        elif kind == "fock":
            c = {"kind": kind, "mesh": ms, "n_ao": n_ao, "n_emb": n}
            cap = 1e12
        elif kind == "bath":
            if nk < 2:
                continue
            c = {"kind": kind, "mesh": ms, "n_ao": n_ao, "n_val": rng.randint(max(1, n_ao // 2), n_ao)}
            cap = 1e12
        elif kind == "fftdf":
            mesh = rng.choice([(1, 1, 1), (2, 1, 1), (2, 2, 1), (2, 2, 2)])
            c = {"kind": kind, "mesh": "x".join(map(str, mesh)), "n_ao": _log(rng, 2, 10), "grid": rng.choice([6, 8, 9, 10, 12]),
                 "n_emb": _log(rng, 4, 18)}
            if c["n_emb"] > math.prod(mesh) * c["n_ao"]:
                continue
            cap = 0.02e12
        else:
            lo = rng.randint(4, 8)
            c = {"kind": "batch", "n_problems": rng.randint(3, 16), "shapes": rng.randint(1, 1 << 20), "n_ao_min": lo,
                 "n_ao_max": lo + rng.randint(2, 6), "n_emb_min": 8, "n_emb_max": rng.randint(24, 56),
                 "prec": rng.choice(["bf16x3", "bf16x3", "fp16x2"])}
            cap = 1e12
        w = work(c)
        full_l = 16 * nk * nk * n_aux * n_ao * n_ao if kind not in ("jk", "fock", "bath", "fftdf", "batch") else 0
        if w["flops"] <= cap and w["bytes"] <= 4e9 and full_l <= 8e9:
            return c


# ---- sizes -------------------------------------------------------------------------------------------------------


def _mesh(case):
    return tuple(int(x) for x in case["mesh"].split("x"))


def _points(mesh):
    g = np.stack(np.meshgrid(*[np.arange(n) for n in mesh], indexing="ij"), -1)
    return g.reshape(-1, 3)


def _index(t, mesh):
    t = np.mod(t, np.asarray(mesh))
    return (t[..., 0] * mesh[1] + t[..., 1]) * mesh[2] + t[..., 2]


def _neg(mesh):
    return _index(-_points(mesh), mesh)


def _add(mesh):
    """[q][k] -> k + q."""
    p = _points(mesh)
    return _index(p[:, None, :] + p[None, :, :], mesh)


def _real_pairs(mesh):
    """(pairs transformed, real K rows per aux function of the contraction) with time reversal: one q of {q, -q}, one
    k1 of {k1, -k1-q}; the factors of q = -q are real."""
    neg, add = _neg(mesh), _add(mesh)
    pairs = rows = 0
    for q in range(len(neg)):
        if q > neg[q]:
            continue
        rows += 1 if q == neg[q] else 2
        pairs += sum(1 for k in range(len(neg)) if k <= neg[add[q][k]])
    return pairs, rows


def _batch_shapes(case):
    """Sizes of the batch's problems: Nk from {8, 27, 36, 64}, n_AO and n_emb uniform, every other one unrestricted."""
    r = np.random.Generator(np.random.Philox(key=[int(case["shapes"]), 77]))
    meshes = {8: (2, 2, 2), 27: (3, 3, 3), 36: (6, 6, 1), 64: (4, 4, 4)}
    out = []
    for p in range(case["n_problems"]):
        mesh = meshes[int(r.choice([8, 27, 36, 64]))]
        n_ao = int(r.integers(case["n_ao_min"], case["n_ao_max"] + 1))
        n = int(r.integers(case["n_emb_min"], min(case["n_emb_max"], math.prod(mesh) * n_ao) + 1))
        out.append(_eri(None, mesh, n_ao, int(8.5 * n_ao + 0.5), n, case["prec"], n if p % 2 else 0, decay=0.7))
    return out


def _spins(case):
    return [case["n_emb"]] + ([case["n_emb_b"]] if case.get("n_emb_b") else [])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [work(c) for c in _batch_shapes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    mesh = _mesh(case)
    nk = math.prod(mesh)
    na, nx, n = case.get("n_ao", 0), case.get("n_aux", 0), case.get("n_emb", 0)
    if kind in ("eri", "three_index"):
        real = case.get("orbitals", "real") == "real"
        pairs, rows = _real_pairs(mesh) if real else (nk * nk, 2 * nk)
        nb = 16.0 * (pairs * nx * na * na + sum(nk * na * s for s in _spins(case)))
        fl = sum(8.0 * pairs * nx * (na * na * s + na * s * s) for s in _spins(case))
        if kind == "three_index":
            return {"bytes": nb + 16.0 * nk * nx * n * n, "flops": fl}
        if real:
            np_ = [s * (s + 1) // 2 for s in _spins(case)]
            same = sum(p * (p + 1.0) for p in np_)
            cross = 2.0 * np_[0] * np_[1] if len(np_) == 2 else 0.0
            return {"bytes": nb + 4.0 * (same + cross), "flops": fl + rows * nx * (same + cross)}
        return {"bytes": nb + 16.0 * n ** 4, "flops": fl + 4.0 * n ** 4 * nk * nx}  # (kl|ij) = (ij|kl)
    if kind == "jk":
        return {"bytes": 16.0 * nk * nx * n * n + 48.0 * n * n, "flops": 16.0 * nk * nx * (n ** 3 + n * n)}
    if kind == "fock":
        np_ = n * (n + 1) // 2
        return {"bytes": 4.0 * np_ * (np_ + 1.0) + 16.0 * nk * na * (na + n) + 16.0 * n * n,
                "flops": 8.0 * nk * (na * na * n + na * n * n) + 4.0 * n ** 4}
    if kind == "bath":
        nv = case["n_val"]
        return {"bytes": 16.0 * nk * na * (2 * na + na + nv),
                "flops": 8.0 * nk * nk * na * nv + 4.0 * (nk - 1) * na * nv * nv + 8.0 * nk * na * na * (na + nv)}
    ng = case["grid"] ** 3
    dft = nk * n * n * ng * 5.0 * math.log2(ng) * 2
    return {"bytes": 16.0 * (nk * nk * ng * na * na + nk * na * n + n ** 4),
            "flops": 8.0 * nk * nk * ng * (na * na * n + na * n * n) + dft + 8.0 * nk * ng * n ** 4}


# ---- inputs ------------------------------------------------------------------------------------------------------


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFF)
    return g


def _normal(shape, g):
    return torch.randn(shape, dtype=F64, device="cuda", generator=g)


def _norms(mesh):
    """|R| of each cell, minimum image."""
    m, n = _points(mesh).astype(float), np.asarray(mesh, dtype=float)
    m = np.where(m > n / 2, m - n, m)
    return torch.from_numpy(np.sqrt((m * m).sum(-1))).cuda()


def _phases(mesh):
    """exp(-i k.R) [k][R]."""
    p, n = _points(mesh).astype(float), np.asarray(mesh, dtype=float)
    return torch.from_numpy(np.exp(-2j * np.pi * (p[:, None, :] * p[None, :, :] / n).sum(-1))).cuda()


def _make_l(case, seed, pairs=None):
    """L[k1][k2][P][mu][nu], or its blocks `pairs`: the Fourier transform of a real tensor B[P][mu R1][nu R2] that is
    symmetric under (mu, R1) <-> (nu, R2) and decays with |R1| + |R2|."""
    mesh, na, nx = _mesh(case), case["n_ao"], case["n_aux"]
    nk = math.prod(mesh)
    w = torch.exp(-case.get("decay", 0.6) * _norms(mesh))
    g = _gen(seed, 1)
    out = torch.empty((nk, nk, nx, na, na) if pairs is None else (len(pairs), nx, na, na), dtype=C128, device="cuda")
    if pairs is not None:
        k1, k2 = (torch.from_numpy(x).cuda() for x in (pairs // nk, pairs % nk))
    step = max(1, int(1.5e8 / (na * nk) ** 2))
    for p0 in range(0, nx, step):
        np_ = min(step, nx - p0)
        b = _normal((np_, na, nk, na, nk), g)
        b *= w[None, None, :, None, None] * w
        b = 0.5 * (b + b.permute(0, 3, 4, 1, 2))
        f = torch.fft.fftn(b.reshape(np_, na, *mesh, na, nk), dim=(2, 3, 4))
        f = torch.fft.ifftn(f.reshape(np_, na, nk, na, *mesh), dim=(4, 5, 6), norm="forward")
        f = f.reshape(np_, na, nk, na, nk).permute(2, 4, 0, 1, 3)
        if pairs is None:
            out[:, :, p0:p0 + np_] = f
        else:
            out[:, p0:p0 + np_] = f[k1, k2]
    return out


def _orthonormal(a):
    q, r = torch.linalg.qr(a)
    d = torch.diagonal(r)
    return q * torch.where(d.abs() > 0, d / d.abs(), torch.ones_like(d)).conj()


def _make_c(case, seed, spin=0):
    """Bloch sums C[k][mu][i] of orthonormal supercell orbitals."""
    mesh, na, n = _mesh(case), case["n_ao"], _spins(case)[spin]
    nk = math.prod(mesh)
    g = _gen(seed, 2 + spin)
    a = _normal((nk, na, n), g)
    if case.get("orbitals") == "complex":
        a = torch.complex(a, _normal((nk, na, n), g))
    a = a * torch.exp(-case.get("decay", 0.6) * _norms(mesh))[:, None, None]
    if case.get("log_range"):
        a = a * 10.0 ** (-case["log_range"] * torch.rand((nk, na, n), dtype=F64, device="cuda", generator=g))
    csc = _orthonormal(a.reshape(nk * na, n)).to(C128).reshape(nk, na * n)
    return (_phases(mesh) @ csc).view(nk, na, n).contiguous()


def _make_density(n, seed):
    """Spin-summed density [n][n] with occupations in [0, 2]."""
    g = _gen(seed, 5)
    q = _orthonormal(_normal((n, n), g))
    occ = 2.0 * torch.rand(n, dtype=F64, device="cuda", generator=g)
    occ[: n // 2] = 2.0
    return ((q * occ) @ q.T).contiguous()


def _real_space_k(mesh, na, seed, stream, antisymmetric=False, decay=0.6):
    """x[k] = sum_R exp(+i k.R) x(R) of a real x(R) that decays, with x(-R) = +-x(R)^T."""
    nk = math.prod(mesh)
    x = _normal((nk, na, na), _gen(seed, stream)) * torch.exp(-decay * _norms(mesh))[:, None, None]
    xt = x[torch.from_numpy(_neg(mesh)).cuda()].transpose(1, 2)
    x = 0.5 * (x - xt if antisymmetric else x + xt)
    return (_phases(mesh).conj() @ x.to(C128).reshape(nk, na * na)).view(nk, na, na)


def _make_bath(case, seed):
    """(gamma^k of a gapped mean field, C^{k,AO,LO} unitary, valence LOs)."""
    mesh, na = _mesh(case), case["n_ao"]
    nk = math.prod(mesh)
    n_occ = max(1, na // 2)
    h = _real_space_k(mesh, na, seed, 6)
    h = 0.9 * h / torch.linalg.matrix_norm(h, 2).max()
    g = _gen(seed, 7)
    order = torch.randperm(na, device="cuda", generator=g)
    eps = torch.ones(na, dtype=F64, device="cuda")
    eps[order[:n_occ]] = -1.0
    _, v = torch.linalg.eigh(h + torch.diag(eps).to(C128))
    occ = v[:, :, :n_occ]
    gamma = (occ @ occ.mH).contiguous()
    x = 0.5 * _real_space_k(mesh, na, seed, 8, antisymmetric=True)
    eye = torch.eye(na, dtype=C128, device="cuda")
    c_lo = torch.linalg.solve(eye + x, eye - x)  # Cayley transform: unitary, time-reversal symmetric
    val = sorted(torch.randperm(na, device="cuda", generator=g)[: case["n_val"]].tolist())
    return gamma, c_lo.contiguous(), val


def _make_factors(case, seed):
    """L^q_P [q][P][i][j] of real orbitals: symmetric in ij, L^{-q} = conj L^q, smaller for later aux functions."""
    mesh, nx, n = _mesh(case), case["n_aux"], case["n_emb"]
    nk = math.prod(mesh)
    g = _gen(seed, 9)
    neg = _neg(mesh)
    out = torch.empty((nk, nx, n, n), dtype=C128, device="cuda")
    scale = torch.exp(-2.0 * torch.arange(nx, dtype=F64, device="cuda") / nx)[:, None, None]
    for q in range(nk):
        if q > neg[q]:
            continue
        re, im = _normal((nx, n, n), g), _normal((nx, n, n), g)
        if q == neg[q]:
            im.zero_()
        x = torch.complex(re + re.transpose(1, 2), im + im.transpose(1, 2)) * scale
        out[q] = x
        out[int(neg[q])] = x.conj()
    return out


_LATTICE = ((2.0, 0.0, 0.0), (0.3, 2.2, 0.0), (0.1, 0.2, 2.5))


def _make_fftdf(case, seed):
    """(rho[k1][k2][r][mu][nu], C): Gaussian AOs on the cell grid, their Bloch sums and pair densities."""
    mesh, na, gr = _mesh(case), case["n_ao"], case["grid"]
    n3 = torch.tensor(mesh, dtype=F64, device="cuda")
    g = _gen(seed, 10)
    centres = torch.rand((na, 3), dtype=F64, device="cuda", generator=g)
    alphas = 1.5 + 1.5 * torch.rand(na, dtype=F64, device="cuda", generator=g)
    frac = torch.from_numpy(_points((gr, gr, gr)) / gr).cuda()
    cells = torch.from_numpy(_points(mesh).astype(float)).cuda()
    d = frac[None, None] - cells[:, None, None] - centres[None, :, None]
    d -= n3 * torch.round(d / n3)
    x = d @ torch.tensor(_LATTICE, dtype=F64, device="cuda")
    chi = torch.exp(-alphas[None, :, None] * (x * x).sum(-1))                     # [R][mu][r]
    nk = math.prod(mesh)
    phi = (_phases(mesh).conj() @ chi.to(C128).reshape(nk, -1)).view(nk, na, -1)     # [k][mu][r]
    rho = torch.einsum("amr,bnr->abrmn", phi.conj(), phi).contiguous()
    return rho, _make_c(dict(case, decay=0.0), seed)


def _desc(case, layout=0):
    ns = _spins(case)
    real = case.get("orbitals", "real") == "real"
    return dm.make_desc(_mesh(case), case["n_ao"], case["n_aux"], ns if len(ns) == 2 else ns[0], n_spin=len(ns),
                        prec=PREC[case["prec"]], sym=B.DMET_SYM_REAL if real else B.DMET_SYM_NONE, l_layout=layout)


class _State:
    """Inputs, output buffers and the plan that a program keeps; the plan goes with it."""

    def __init__(self, case, descs, workspace=0):
        self.kind = case["kind"]
        self.plan = dm.dmet_emb_plan(descs, stream=torch.cuda.current_stream().cuda_stream, workspace_limit=workspace)

    def __del__(self):
        if getattr(self, "plan", None):
            dm.dmet_emb_destroy(self.plan)


def _eri_inputs(case, seed):
    """(descriptor, L as the call takes it, orbitals per spin)."""
    desc = _desc(case, B.DMET_L_REDUCED if case["reduced"] else B.DMET_L_FULL)
    pairs = np.asarray(dm.dmet_emb_l_pairs(desc)).astype(np.int64) if case["reduced"] else None
    return desc, _make_l(case, seed, pairs), [_make_c(case, seed, s) for s in range(desc.n_spin)]


def _eri_outputs(desc):
    full = desc.sym == B.DMET_SYM_NONE
    return [torch.empty(dm.dmet_emb_eri_bytes(desc, b) // (16 if full else 8), dtype=C128 if full else F64, device="cuda")
            for b in range(1 if desc.n_spin == 1 else 3)]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("eri", "batch"):
        probs = [_eri_inputs(c, seed * 100 + i) for i, c in enumerate(_batch_shapes(case))] if kind == "batch" \
            else [_eri_inputs(case, seed)]
        s = _State(case, [p[0] for p in probs], (32 << 30) if kind == "batch" else 0)
        s.L, s.C = [p[1] for p in probs], [p[2] for p in probs]
        s.out = [_eri_outputs(p[0]) for p in probs]
        if kind == "batch":
            dm.dmet_emb_graph(s.plan, True)
        return s
    mesh = _mesh(case)
    nk, na, n = math.prod(mesh), case.get("n_ao", 1), case.get("n_emb", 0)
    if kind == "three_index":
        s = _State(case, _desc(case))
        s.L, s.C, s.nk = _make_l(case, seed), _make_c(case, seed), nk
        s.out = torch.empty((nk, case["n_aux"], n, n), dtype=C128, device="cuda")
    elif kind == "jk":
        s = _State(case, dm.make_desc(mesh, n, case["n_aux"], n))  # n_AO does not enter this call
        s.Lq, s.gamma = _make_factors(case, seed), _make_density(n, seed).to(C128)
        s.out = [torch.empty((n, n), dtype=C128, device="cuda") for _ in range(2)]
    elif kind == "fock":
        s = _State(case, dm.make_desc(mesh, na, 1, n))
        s.F, s.C, s.gamma = _real_space_k(mesh, na, seed, 11).contiguous(), _make_c(case, seed), _make_density(n, seed)
        s.eri, s.out = _packed_eri(n, seed)[0], torch.empty((n, n), dtype=F64, device="cuda")
    elif kind == "bath":
        s = _State(case, dm.make_desc(mesh, na, 1, na + case["n_val"]))
        s.gamma, s.C_lo, s.val = _make_bath(case, seed)
        s.out = torch.empty((nk, na, na + case["n_val"]), dtype=C128, device="cuda")
    else:
        gr = case["grid"]
        s = _State(case, dm.make_desc(mesh, na, gr ** 3, n, eri_pack=B.DMET_PACK_FULL), 16 << 30)
        s.rho, s.C = _make_fftdf(case, seed)
        s.grid, s.out = (gr, gr, gr), torch.empty(n ** 4, dtype=C128, device="cuda")
    return s


def run(s):
    if s.kind in ("eri", "batch"):
        dm.dmet_emb_eri(s.plan, s.L, s.C, s.out)
    elif s.kind == "three_index":
        dm.dmet_emb_transform_3idx(s.plan, 0, s.L, [s.C], 0, s.nk, [s.out])
    elif s.kind == "jk":
        dm.dmet_emb_jk_df(s.plan, s.Lq, s.gamma, *s.out)
    elif s.kind == "fock":
        dm.dmet_emb_fock(s.plan, s.F, s.C, s.eri, s.gamma, s.out)
    elif s.kind == "bath":
        dm.dmet_emb_bath(s.plan, s.gamma, s.C_lo, s.val, s.out)
    else:
        dm.dmet_emb_eri_fftdf(s.plan, s.rho, [s.C], s.grid, _LATTICE, [s.out])
    return s.out


# ---- the same in plain torch, 64 bits ----------------------------------------------------------------------------


def _factors(L, C, mesh):
    """L^q_{P,ij} = (1/Nk) sum_k1 C^{k1+} L^{k1,k1+q}_P C^{k1+q}, [q][P][i][j]."""
    nk, nx, na, n = L.shape[0], L.shape[2], C.shape[1], C.shape[2]
    add = torch.from_numpy(_add(mesh)).cuda()
    bra = C.reshape(nk * na, n).mH.contiguous()                                    # [i][(k1 mu)]
    out = torch.empty((nk, nx, n, n), dtype=C128, device="cuda")
    ks = torch.arange(nk, device="cuda")
    step = max(1, int(2e8 / (nk * na * max(n, na))))
    for q in range(nk):
        for p0 in range(0, nx, step):
            b = L[ks, add[q], p0:p0 + step]                                       # [k1][P][mu][nu]
            m = b.shape[1]
            t = torch.bmm(b.reshape(nk, m * na, na), C[add[q]]).view(nk, m, na, n)
            t = t.permute(1, 0, 2, 3).reshape(m, nk * na, n)
            out[q, p0:p0 + m] = torch.matmul(bra, t) / nk
    return out


def _tri(n):
    i, j = np.tril_indices(n)
    return torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda()


def _exact_eri(case, seed):
    mesh = _mesh(case)
    nk = math.prod(mesh)
    neg = torch.from_numpy(_neg(mesh)).cuda()
    L = _make_l(case, seed)
    lq = [_factors(L, _make_c(case, seed, s), mesh) for s in range(len(_spins(case)))]
    del L
    if case["orbitals"] == "complex":
        a = lq[0].flatten(0, 1).flatten(1)
        b = lq[0][neg].flatten(0, 1).flatten(1)
        return [(a.T @ b / nk).reshape(-1)]
    out = []
    pk = []
    for x in lq:
        i, j = _tri(x.shape[2])
        pk.append(x[:, :, i, j])                                                 # [q][P][i >= j]
    for s in range(len(pk)):
        for t in range(s, len(pk)):
            a, b = pk[s].flatten(0, 1), pk[t][neg].flatten(0, 1)
            e = (a.real.contiguous().T @ b.real.contiguous() - a.imag.contiguous().T @ b.imag.contiguous()) / nk
            if s == t:
                i, j = _tri(e.shape[0])
                e = e[i, j]
            out.append(e.reshape(-1))
    return out


def _packed_eri(n, seed):
    """(8-fold packed, dense over pairs) ERI: a sum of outer products over the pairs ij."""
    np_ = n * (n + 1) // 2
    r = min(np_, 400)
    x = _normal((r, np_), _gen(seed, 12)) / math.sqrt(r)
    e = x.T @ x
    i, j = _tri(np_)
    return e[i, j].contiguous(), e


def _exact_fftdf(case, seed):
    mesh, gr, n = _mesh(case), case["grid"], case["n_emb"]
    rho, C = _make_fftdf(case, seed)
    nk, ng = math.prod(mesh), gr ** 3
    lq = _factors(rho, C, mesh)                                                   # [q][r][i][j]
    lat = np.asarray(_LATTICE)
    omega, recip = abs(np.linalg.det(lat)), 2.0 * np.pi * np.linalg.inv(lat).T
    pts, neg, frac = _points(mesh), _neg(mesh), _points((gr, gr, gr)) / gr
    eri = torch.zeros((n * n, n * n), dtype=C128, device="cuda")
    for q in range(nk):
        t = pts[q] / np.asarray(mesh)
        ph = torch.from_numpy(np.exp(-2j * np.pi * (frac @ t))).cuda()[:, None, None]
        axes = []
        for d in range(3):  # the supercell's signed FFT frequency of each plane wave: n + N m with m = j mod g
            big = mesh[d] * gr
            f = pts[q][d] + mesh[d] * np.arange(gr)
            axes.append(np.where(f >= (big + 1) // 2, f - big, f) / mesh[d])
        v = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3) @ recip
        g2 = (v * v).sum(-1)
        ker = torch.from_numpy(np.where(g2 > 1e-12, 4.0 * np.pi / np.where(g2 > 1e-12, g2, 1.0), 0.0)).cuda()
        hat = torch.fft.fftn((ph * lq[q]).view(gr, gr, gr, n, n), dim=(0, 1, 2)) * ker.view(gr, gr, gr, 1, 1)
        w = torch.fft.ifftn(hat, dim=(0, 1, 2)).reshape(ng, n, n) * ph.conj()
        eri += omega / ng / nk * (w.reshape(ng, n * n).T @ lq[int(neg[q])].reshape(ng, n * n))
    return eri.reshape(-1)


def _exact_bath(case, seed):
    mesh, na = _mesh(case), case["n_ao"]
    nk = math.prod(mesh)
    gamma, c_lo, val = _make_bath(case, seed)
    e = _phases(mesh)
    block = (e.conj().T @ gamma.reshape(nk, na * na)).view(nk, na, na)[1:, :, val].real / nk
    u = torch.linalg.svd(block.reshape((nk - 1) * na, len(val)), full_matrices=False)[0]
    at = u.abs().argmax(0)
    u = u * torch.sign(u.gather(0, at[None]))
    c = torch.zeros((nk, na, na + len(val)), dtype=C128, device="cuda")
    c[0, :, :na] = torch.eye(na, dtype=C128, device="cuda")
    c[1:, :, na:] = u.view(nk - 1, na, len(val)).to(C128)
    return c_lo @ (e @ c.view(nk, -1)).view(c.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_exact_eri(c, seed * 100 + i) for i, c in enumerate(_batch_shapes(case))]
    if kind == "eri":
        # above this the dense sums take more than some twenty seconds
        return None if work(case)["flops"] > 8e12 else [_exact_eri(case, seed)]
    mesh = _mesh(case)
    nk = math.prod(mesh)
    if kind == "three_index":
        return _factors(_make_l(case, seed), _make_c(case, seed), mesh)
    if kind == "jk":
        lq, gamma = _make_factors(case, seed), _make_density(case["n_emb"], seed).to(C128)
        m = lq[torch.from_numpy(_neg(mesh)).cuda()]
        tr = torch.einsum("qpkl,lk->qp", m, gamma)
        n = gamma.shape[0]
        j = (tr.reshape(1, -1) @ lq.view(-1, n * n)).view(n, n) / nk
        k = torch.zeros_like(gamma)
        for q in range(nk):
            x = (lq[q] @ gamma).permute(1, 0, 2).reshape(n, -1)                   # [i][(P l)]
            k += x @ m[q].reshape(-1, n) / nk
        return [j, k]
    if kind == "fock":
        n = case["n_emb"]
        F, C, gamma = _real_space_k(mesh, case["n_ao"], seed, 11), _make_c(case, seed), _make_density(n, seed)
        f0 = (C.mH @ F @ C).sum(0).real / nk
        e = _packed_eri(n, seed)[1]
        i, j = _tri(n)
        pair = torch.empty((n, n), dtype=torch.long, device="cuda")
        pair[i, j] = pair[j, i] = torch.arange(len(i), device="cuda")
        jm = (e[pair.reshape(-1)][:, pair.reshape(-1)] @ gamma.T.reshape(-1)).view(n, n) if n <= 64 else \
            (e @ torch.where(i == j, gamma[i, j], gamma[i, j] + gamma[j, i]))[pair]
        km = torch.empty_like(gamma)
        for a in range(n):
            km[a] = torch.einsum("klj,kl->j", e[pair[a]][:, pair], gamma)          # (a k | l j) gamma_kl
        return f0 - (jm - 0.5 * km)
    return _exact_bath(case, seed) if kind == "bath" else _exact_fftdf(case, seed)

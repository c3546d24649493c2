"""FP64 products through residues (csrc/rns.cu) at the sizes where they can go wrong: odd rows and columns, K that
is no multiple of a K block, K of several accumulation segments, several chunks under a small workspace limit, the
rectangular alpha-beta block, complex orbitals with dense and 4-fold packed output, wide dynamic range, and
non-finite inputs, through the public entry points against the oracle.

Bound: every step rounds its operands to 2^-58 of a row's norm and its results to 2^-53, and the three steps
(two half transforms, contraction) each add a few such roundings, so results agree to a few 1e-15 of the largest;
the oracle's own FP64 sums over up to some 1e4 terms carry about 2^-53 sqrt(1e4) = 1e-14. 1e-13 holds both."""
import numpy as np
import pytest

import oracle
from oracle.checks import pack_s4
import synth
import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import out_buffers, run_3idx, run_eri, torch_cuda

pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def check(got, ref):
    ref = np.ravel(ref)
    assert np.abs(got - ref).max() < TOL * np.abs(ref).max(), np.abs(got - ref).max() / np.abs(ref).max()


# (mesh, n_ao, n_aux, n_emb): odd everything; K just past one K block; a contraction of more than 960 K
# (two segments); one cell; 128 and 129 pairs of columns
CASES = [((3, 2, 1), 13, 67, 37), ((2, 2, 1), 33, 129, 31), ((3, 3, 1), 9, 131, 45), ((1, 1, 1), 47, 403, 33),
         ((2, 2, 2), 16, 128, 64)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])) + f"_{c[1]}_{c[2]}_{c[3]}")
@pytest.mark.parametrize("limit", [0, 48 << 20])
def test_packed(torch, case, limit):
    mesh, nao, naux, n = case
    spec = synth.LatticeSpec(mesh, nao, naux, n, 1, 0.6, 0.0, 71, "r")
    L, (C,), _ = synth.make_problem(spec)
    (got,), st, _ = run_eri(torch, B.make_desc(mesh, nao, naux, n), L, [C], workspace_limit=limit)
    assert st == B.DMET_OK
    check(got, oracle.pack_s8(oracle.embedded_eri(L, C, mesh).real))


def test_unrestricted_log_range(torch):
    """n_alpha != n_beta, orbital coefficients over four decades, L rows scaled over twelve."""
    spec = synth.LatticeSpec((3, 2, 1), 14, 83, 41, 2, 0.6, 4.0, 72, "r")
    spec_b = synth.spec_with(spec, n_emb=38)
    L = synth.make_L(spec)
    L = L * (10.0 ** np.linspace(-6, 6, spec.n_aux))[None, None, :, None, None]
    Ca = synth.bloch_orbitals(synth.supercell_orbitals(spec, 0), spec.mesh)
    Cb = synth.bloch_orbitals(synth.supercell_orbitals(spec_b, 1), spec.mesh)
    got, st, _ = run_eri(torch, B.make_desc(spec.mesh, 14, 83, [41, 38], n_spin=2), L, [Ca, Cb])
    assert st == B.DMET_OK
    check(got[0], oracle.pack_s8(oracle.embedded_eri(L, Ca, spec.mesh).real))
    check(got[2], oracle.pack_s8(oracle.embedded_eri(L, Cb, spec.mesh).real))
    ab = oracle.embedded_eri(L, Ca, spec.mesh, Cb).real
    ia, ib = np.tril_indices(41), np.tril_indices(38)
    check(got[1], ab[ia[0], ia[1]][:, ib[0], ib[1]])


@pytest.mark.parametrize("pack", [B.DMET_PACK_FULL, B.DMET_PACK_S4])
def test_complex_orbitals(torch, pack):
    spec = synth.LatticeSpec((3, 2, 1), 11, 61, 19, 1, 0.6, 0.0, 73, "r")
    L = synth.make_L(spec)
    C = synth.bloch_orbitals(synth.complex_supercell_orbitals(spec), spec.mesh)
    d = B.make_desc(spec.mesh, 11, 61, 19, sym=B.DMET_SYM_NONE, eri_pack=pack)
    (got,), st, _ = run_eri(torch, d, L, [C])
    assert st == B.DMET_OK
    ref = oracle.embedded_eri(L, C, spec.mesh)
    got = got.view(np.complex128) if got.dtype != np.complex128 else got
    check(got, ref if pack == B.DMET_PACK_FULL else pack_s4(ref))


def test_three_index(torch):
    spec = synth.LatticeSpec((3, 2, 1), 17, 90, 35, 1, 0.6, 0.0, 74, "r")
    L, (C,), _ = synth.make_problem(spec)
    (got,), st, _ = run_3idx(torch, B.make_desc(spec.mesh, 17, 90, 35), L, [C], 0, 6)
    assert st == B.DMET_OK
    check(got.ravel(), oracle.embedded_3idx(L, C, spec.mesh))


def test_non_finite_and_tiny(torch):
    """A NaN in one aux function's L reaches every result (each sums over it); magnitudes near the ends of the
    exponent range scale through."""
    spec = synth.LatticeSpec((2, 2, 1), 20, 99, 40, 1, 0.6, 0.0, 75, "r")
    L, (C,), _ = synth.make_problem(spec)
    d = B.make_desc(spec.mesh, 20, 99, 40)
    ref = oracle.pack_s8(oracle.embedded_eri(L, C, spec.mesh).real)
    for s in (2.0 ** -500, 2.0 ** 480):
        (got,), _, _ = run_eri(torch, d, L * s, [C])
        check(got / s / s, ref)
    bad = L.copy()
    bad[0, 0, 5, 3, 4] = np.nan
    (got,), _, _ = run_eri(torch, d, bad, [C])
    assert np.isnan(got).all()


@pytest.mark.parametrize("mesh,n_aux,n,real", [((3, 2, 1), 91, 37, True), ((2, 2, 1), 130, 64, False), ((3, 1, 1), 53, 131, True)])
def test_coulomb_exchange_from_factors(torch, mesh, n_aux, n, real):
    """dmet_emb_jk_df in chunks of q with K split into ragged parts of the aux functions; factors without any
    symmetry between q and -q."""
    nk = int(np.prod(mesh))
    rng = np.random.default_rng(6)
    Lq = rng.standard_normal((nk, n_aux, n, n)) + 1j * rng.standard_normal((nk, n_aux, n, n))
    gamma = synth.embedding_density(n, 9).astype(np.complex128)
    if not real:
        gamma = gamma + 0.1j * rng.standard_normal((n, n))
    d = dm.make_desc(mesh, max(1, -(-n // nk)), n_aux, n, sym=B.DMET_SYM_NONE)
    Ld, gd = torch.from_numpy(Lq).cuda(), torch.from_numpy(gamma).cuda()
    J = torch.empty((n, n), dtype=torch.complex128, device="cuda")
    K = torch.empty_like(J)
    plan = dm.dmet_emb_plan(d, stream=torch.cuda.current_stream().cuda_stream)
    try:
        for _ in range(2):
            dm.dmet_emb_jk_df(plan, Ld, gd, J, K)
        st, _ = dm.dmet_emb_status(plan, 0)
    finally:
        dm.dmet_emb_destroy(plan)
    assert st == B.DMET_OK
    Jr, Kr = oracle.coulomb_exchange_df(Lq, gamma, mesh)
    check(J.cpu().numpy().ravel(), Jr)
    check(K.cpu().numpy().ravel(), Kr)


@pytest.mark.parametrize("n_aux", [60, 700])
def test_expired_waits(torch, n_aux):
    """The residue GEMM's bounded waits, alone and with its CTAs in clusters (the longer products): with the copies
    withheld they give up after 2 ms, the status says so once, and the same plan then runs normally."""
    spec = synth.LatticeSpec((3, 2, 1), 24, n_aux, 48, 1, 0.6, 0.0, 76, "r")
    L, (C,), _ = synth.make_problem(spec)
    d = B.make_desc(spec.mesh, 24, n_aux, 48)
    Ld, Cd = torch.from_numpy(L).cuda(), torch.from_numpy(C).cuda()
    outs = out_buffers(torch, d)
    plan = dm.dmet_emb_plan(d, stream=torch.cuda.current_stream().cuda_stream)
    try:
        dm.dmet_emb_wait_limit(plan, 2_000_000, test_withhold_loads=True)
        dm.dmet_emb_eri(plan, [Ld], [[Cd]], [outs])
        st, _ = dm.dmet_emb_status(plan, 0)
        assert st == B.DMET_ERR_TIMEOUT
        dm.dmet_emb_wait_limit(plan, 0)
        dm.dmet_emb_eri(plan, [Ld], [[Cd]], [outs])
        st, _ = dm.dmet_emb_status(plan, 0)
        assert st == B.DMET_OK
    finally:
        dm.dmet_emb_destroy(plan)
    check(outs[0].cpu().numpy(), oracle.pack_s8(oracle.embedded_eri(L, C, spec.mesh).real))

"""The kernels that sort the transformed integrals into the contraction's operand, at the edges of their tiles: 8 x 8
blocks of pairs by 32 auxiliary functions for real embedding orbitals, 16 orbitals by 64 auxiliary functions for complex
ones, with both widths of their stores (odd numbers of auxiliary functions take the narrow one) and both element sizes.
Tolerance, as for the other shapes of these precisions: 1e-6 relative Frobenius norm and max-abs over max for three BF16
slices (24 bits), 5e-6 for the 22-bit ones."""
import numpy as np
import pytest

import oracle
import synth
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import rel_fro, run_eri, torch_cuda
from test_gpu_mixed_complex import run as run_complex

pytestmark = pytest.mark.gpu

PRECS = [("bf16x3", B.DMET_PREC_BF16X3, 1e-6), ("fp16x2", B.DMET_PREC_FP16X2, 5e-6), ("tf32x3", B.DMET_PREC_TF32X3, 5e-6)]


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def check(got, ref, tol):
    got = got.reshape(ref.shape)
    assert np.isfinite(got).all()
    e, m = rel_fro(got, ref), np.abs(got - ref).max() / np.abs(ref).max()
    assert e < tol and m < tol, (e, m)


@pytest.mark.parametrize("prec", PRECS, ids=lambda p: p[0])
@pytest.mark.parametrize("mesh,naux,n", [((2, 1, 1), 31, 7), ((2, 1, 1), 33, 8), ((3, 1, 1), 32, 9), ((3, 1, 1), 33, 17),
                                         ((4, 1, 1), 65, 16)], ids=str)
def test_real_orbitals(torch, prec, mesh, naux, n):
    _, p, tol = prec
    spec = synth.LatticeSpec(mesh, 6, naux, n, 1, 0.6, 0.0, 83, "pe")
    L, Cs, _ = synth.make_problem(spec)
    d = B.make_desc(mesh, 6, naux, [n, 0], prec=p)
    (got,), st, stats = run_eri(torch, d, L, Cs)
    assert st == B.DMET_OK, (st, stats)
    check(got, oracle.pack_s8(oracle.embedded_eri(L, Cs[0], spec.mesh).real), tol)


@pytest.mark.parametrize("prec", PRECS, ids=lambda p: p[0])
@pytest.mark.parametrize("mesh,naux,n", [((2, 1, 1), 63, 8), ((3, 1, 1), 64, 15), ((3, 1, 1), 65, 16), ((2, 2, 1), 66, 17)],
                         ids=str)
def test_complex_orbitals(torch, prec, mesh, naux, n):
    _, p, tol = prec
    spec = synth.LatticeSpec(mesh, 8, naux, n, 1, 0.6, 0.0, 89, "pe")
    L = synth.make_L(spec)
    C = synth.bloch_orbitals(synth.complex_supercell_orbitals(spec, 0), spec.mesh)
    d = B.make_desc(mesh, 8, naux, n, sym=B.DMET_SYM_NONE, eri_pack=B.DMET_PACK_FULL, prec=p)
    (got,) = run_complex(torch, d, L, [C])
    check(got, oracle.embedded_eri(L, C, spec.mesh), tol)

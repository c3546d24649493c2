"""FP64 results element by element on operands that are graded over far more than FP64's 53 bits: orbitals and integrals
that decay with the distance of their indices, so that most results lie many decades below the norms of the rows that
enter them.

Bound: a sum over K products in FP64, in any order, is off by at most K 2^-53 sum |a_k b_k| (4 K for a complex one, with
moduli); the three-index factors are two such sums, over n_AO and over Nk n_AO terms, and the contraction a third, over
Nk n_aux (twice that for Re and Im). Bounded over the sums of the moduli, which keep the grading, the result and the
reference, plain FP64 as well, each are within c 2^-53 of exact, c the sum of these numbers of terms."""
import numpy as np
import pytest

import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import run_3idx, run_eri, torch_cuda

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def graded(rng, nk, nao, naux, n, decades, real):
    """L[k1][k2][P][mu][nu] and C[k][mu][i] with moduli falling by `decades` over the index distance; every sixth
    aux function touches only the first half of the AOs."""
    mu, i = np.arange(nao), np.arange(n) * (nao / n)
    shape = (nk, nk, naux, nao, nao)
    L = rng.standard_normal(shape) + (0 if real else 1j * rng.standard_normal(shape))
    L = L * 10.0 ** (-decades * np.abs(mu[:, None] - mu[None, :]) / nao)
    L[:, :, ::6, nao // 2:, :] = 0
    L[:, :, ::6, :, nao // 2:] = 0
    if real:
        L = L + L.transpose(1, 0, 2, 4, 3)
    C = rng.standard_normal((nk, nao, n)) + (0 if real else 1j * rng.standard_normal((nk, nao, n)))
    C = C * 10.0 ** (-decades * np.abs(mu[:, None] - i[None, :]) / nao)
    return L.astype(np.complex128), C.astype(np.complex128)


def factors(L, C, dims):
    """L^q_P = (1/Nk) sum_k1 C^{k1+} L^{k1,k1+q}_P C^{k1+q} for C order mesh points."""
    idx = np.stack(np.meshgrid(*[np.arange(d) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    add = np.ravel_multi_index(np.moveaxis((idx[:, None] + idx[None]) % dims, -1, 0), dims)  # [q][k]
    nk = len(idx)
    T = [[L[k, add[q, k]] @ C[add[q, k]] for k in range(nk)] for q in range(nk)]
    return np.stack([sum(C[k].conj().T @ T[q][k] for k in range(nk)) / nk for q in range(nk)]), add


@pytest.mark.parametrize("mesh,nao,naux,n,decades", [((1, 1, 1), 64, 403, 33, 12), ((2, 1, 1), 48, 330, 40, 30),
                                                     ((3, 1, 1), 40, 301, 24, 100), ((1, 1, 1), 96, 257, 64, 0)])
def test_three_index(torch, mesh, nao, naux, n, decades):
    nk = int(np.prod(mesh))
    L, C = graded(np.random.default_rng(decades + n), nk, nao, naux, n, decades, False)
    (got,), _, _ = run_3idx(torch, B.make_desc(mesh, nao, naux, n, sym=B.DMET_SYM_NONE), L, [C], 0, nk)
    ref, _ = factors(L, C, mesh)
    bound, _ = factors(np.abs(L), np.abs(C), mesh)
    err = np.abs(got.reshape(ref.shape) - ref)
    tol = 2 * 4 * (nao + nk * nao + 2) * U * bound
    assert (err <= tol).all(), (err[bound > 0] / (U * bound[bound > 0])).max()


@pytest.mark.parametrize("decades", [0, 12, 40])
def test_packed_eri(torch, decades):
    """One cell, real orbitals: the packed real contraction as well."""
    nao, naux, n = 48, 1100, 32
    L, C = graded(np.random.default_rng(decades), 1, nao, naux, n, decades, True)
    (got,), _, _ = run_eri(torch, B.make_desc((1, 1, 1), nao, naux, n), L, [C])
    i, j = np.tril_indices(n)

    def eri(l, c):
        x = (c.T @ l[0, 0] @ c)[:, i, j]
        return (x.T @ x)[np.tril_indices(len(i))]

    ref, bound = eri(L.real, C[0].real), eri(np.abs(L.real), np.abs(C[0].real))
    tol = 2 * (naux + 2 * 4 * (2 * nao + 2)) * U * bound
    err = np.abs(got - ref)
    assert (err <= tol).all(), (err[bound > 0] / (U * bound[bound > 0])).max()


def test_coulomb_exchange_from_factors(torch):
    """dmet_emb_jk_df with factors graded away from the diagonal and a localised density."""
    n, naux = 72, 150
    rng = np.random.default_rng(5)
    fall = 10.0 ** (-20.0 * np.abs(np.arange(n)[:, None] - np.arange(n)[None]) / n)
    Lq = ((rng.standard_normal((1, naux, n, n)) + 1j * rng.standard_normal((1, naux, n, n))) * fall)
    gamma = (rng.standard_normal((n, n)) * fall).astype(np.complex128)
    plan = dm.dmet_emb_plan(dm.make_desc((1, 1, 1), n, naux, n, sym=B.DMET_SYM_NONE),
                            stream=torch.cuda.current_stream().cuda_stream)
    J, K = (torch.empty((n, n), dtype=torch.complex128, device="cuda") for _ in range(2))
    try:
        dm.dmet_emb_jk_df(plan, torch.from_numpy(Lq).cuda(), torch.from_numpy(gamma).cuda(), J, K)
        torch.cuda.synchronize()
    finally:
        dm.dmet_emb_destroy(plan)

    def exchange(l, g):
        return sum(x @ g @ x for x in l[0])

    tol = 2 * 4 * (n + naux * n + 2) * U * exchange(np.abs(Lq), np.abs(gamma))
    err = np.abs(K.cpu().numpy() - exchange(Lq, gamma))
    assert (err <= tol).all(), (err / tol).max()

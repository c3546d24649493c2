"""Infinities and NaNs in an operand go the way of the FMAs whichever engine forms the products: the same results are
infinite, NaN and finite with the residue products' scratch and without it (a workspace limit that leaves none)."""
import numpy as np
import pytest

import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu
MESH, NAO, NAUX, N = (2, 1, 1), 40, 120, 24


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def factors(torch, L, C, limit):
    d = B.make_desc(MESH, NAO, NAUX, N, sym=B.DMET_SYM_NONE)
    out = torch.empty((2, NAUX, N, N), dtype=torch.complex128, device="cuda")
    plan = dm.dmet_emb_plan(d, stream=torch.cuda.current_stream().cuda_stream, workspace_limit=limit)
    try:
        dm.dmet_emb_transform_3idx(plan, 0, torch.from_numpy(L).cuda(), [torch.from_numpy(C).cuda()], 0, 2, [out])
        torch.cuda.synchronize()
    finally:
        dm.dmet_emb_destroy(plan)
    return out.cpu().numpy()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["L", "C", "L beside zeros"])
def test_same_as_without_residues(torch, value, where):
    rng = np.random.default_rng(3)
    L = rng.standard_normal((2, 2, NAUX, NAO, NAO)) + 1j * rng.standard_normal((2, 2, NAUX, NAO, NAO))
    C = rng.standard_normal((2, NAO, N)) + 1j * rng.standard_normal((2, NAO, N))
    if where == "C":
        C[1, 7, 5] = value
    else:
        L[0, 1, 33, 4, 9] = value
    if where == "L beside zeros":
        C[1, 9, ::2] = 0          # meets the value in half of the columns
        C[1, :, 3] = 0
    got, ref = factors(torch, L, C, 0), factors(torch, L, C, 10 << 20)
    for a, b in ((got.real, ref.real), (got.imag, ref.imag)):
        assert np.array_equal(np.isnan(a), np.isnan(b))
        assert np.array_equal(np.isposinf(a), np.isposinf(b)) and np.array_equal(np.isneginf(a), np.isneginf(b))
        ok = np.isfinite(b)
        # (both are FP64 sums over at most Nk n_AO^2 products of normal numbers)
        assert ok.any() and np.abs(a[ok] - b[ok]).max() < 1e-12 * np.abs(b[ok]).max()
    if np.isinf(value) and where == "L":
        assert np.isinf(ref).any()

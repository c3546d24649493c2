"""dmet_emb_jk_df for more orbitals than its parts were first sized for: the scratch stays at about 1 GiB, and chunks
of some aux functions of one q (the largest case: several chunks per q, the last ones ragged) give the same J and K."""
import numpy as np
import pytest

import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


# chunks of several whole q, of one q each, and of a part of a q
@pytest.mark.parametrize("nk,n_aux,n", [(5, 97, 61), (3, 431, 181), (2, 503, 283)])
def test_scratch_and_values(torch, nk, n_aux, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    Lq = torch.randn((nk, n_aux, n, n), dtype=torch.complex128, device="cuda", generator=g)
    gamma = torch.randn((n, n), dtype=torch.complex128, device="cuda", generator=g)
    J, K = torch.empty_like(gamma), torch.empty_like(gamma)
    d = dm.make_desc((nk, 1, 1), -(-n // nk), n_aux, n, sym=B.DMET_SYM_NONE)
    plan = dm.dmet_emb_plan(d, stream=torch.cuda.current_stream().cuda_stream)
    try:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        dm.dmet_emb_jk_df(plan, Lq, gamma, J, K)
        torch.cuda.synchronize()
        taken = free - torch.cuda.mem_get_info()[0]
    finally:
        dm.dmet_emb_destroy(plan)
    assert taken < 1.1 * 2 ** 30
    neg = [(nk - q) % nk for q in range(nk)]
    k = sum((Lq[q] @ gamma).permute(1, 0, 2).reshape(n, -1) @ Lq[neg[q]].reshape(-1, n) for q in range(nk)) / nk
    tr = torch.einsum("qpkl,lk->qp", Lq[neg], gamma)
    j = (tr.reshape(1, -1) @ Lq.view(-1, n * n)).view(n, n) / nk
    # random operands: sums of up to n_aux n terms, 2^-53 sqrt of that of the largest, in either
    for got, ref in ((J, j), (K, k)):
        assert (got - ref).abs().max() < 1e-13 * ref.abs().max()

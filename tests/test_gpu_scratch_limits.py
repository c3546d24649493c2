"""FP64 products where the workspace limit leaves little residue scratch: what fits runs through it, in chunks, the
rest as FMAs; no call is refused for it."""
import re

import pytest

import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


# the last: the scales of its 2.4 million rows (as of an FFTDF grid) fill the scratch by themselves
@pytest.mark.parametrize("n_aux,n_ao,n", [(300, 40, 40), (7000, 24, 20), (65536, 36, 16)])
@pytest.mark.parametrize("left", [9 << 20, 20 << 20])
def test_three_index(torch, n_aux, n_ao, n, left):
    d = B.make_desc((1, 1, 1), n_ao, n_aux, n, sym=B.DMET_SYM_NONE)
    stream = torch.cuda.current_stream().cuda_stream
    with pytest.raises(B.DmetError) as e:
        dm.dmet_emb_plan(d, stream=stream, workspace_limit=1)
    need = int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))
    g = torch.Generator(device="cuda").manual_seed(n_aux)
    L = torch.randn((n_aux, n_ao, n_ao), dtype=torch.complex128, device="cuda", generator=g)
    C = torch.randn((n_ao, n), dtype=torch.complex128, device="cuda", generator=g)
    out = torch.empty((1, n_aux, n, n), dtype=torch.complex128, device="cuda")
    plan = dm.dmet_emb_plan(d, stream=stream, workspace_limit=need + left)
    try:
        dm.dmet_emb_transform_3idx(plan, 0, L, [C], 0, 1, [out])
        torch.cuda.synchronize()
    finally:
        dm.dmet_emb_destroy(plan)
    ref = C.mH @ (L @ C)
    # sums over n_AO products, twice: a few 1e-15 of the largest
    assert (out[0] - ref).abs().max() < 1e-13 * ref.abs().max()

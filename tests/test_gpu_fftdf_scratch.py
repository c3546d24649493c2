"""dmet_emb_eri_fftdf where the DFTs run as FFTs, in place: one buffer of N_g n^2 complex values per q."""
import numpy as np
import pytest

import synth
import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def test_one_buffer():
    torch = torch_cuda()
    mesh, nao, grid, n = (2, 2, 2), 3, (16, 15, 14), 24
    spec = synth.GridSpec(mesh, nao, grid, n_emb=n, seed=3)
    nk, ng = int(np.prod(mesh)), int(np.prod(grid))
    rho = torch.randn((nk, nk, ng, nao, nao), dtype=torch.complex128, device="cuda")
    C = torch.from_numpy(synth.bloch_orbitals(synth.grid_orbitals(spec), mesh)).cuda()
    out = torch.empty(n ** 4, dtype=torch.complex128, device="cuda")
    d = dm.make_desc(mesh, nao, ng, n, eri_pack=B.DMET_PACK_FULL)
    plan = dm.dmet_emb_plan(d, stream=torch.cuda.current_stream().cuda_stream, workspace_limit=4 << 30)
    try:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        dm.dmet_emb_eri_fftdf(plan, rho, [C], grid, spec.lattice, [out])
        torch.cuda.synchronize()
        taken = free - torch.cuda.mem_get_info()[0]
    finally:
        dm.dmet_emb_destroy(plan)
    # (the tables and the contraction's four partial blocks of 16 n^4 bytes come to a tenth of it)
    assert taken < 1.5 * nk * ng * n * n * 16
    assert torch.isfinite(torch.view_as_real(out)).all()

"""The in-register FFTs of the FFTDF path (csrc/fftdf.cu) for every axis length they take (prime factors 2, 3, 5, 7,
up to 32 points), each as first, middle and last axis (other phases, source tables and strides), and mixed with a length
they do not take (11), which sends the whole grid to the dense passes. Against the oracle, with the
FFTDF bound of 1e-12 of the largest |(ij|kl)|."""
import numpy as np
import pytest

import synth
import oracle.fftdf as of
import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu

LENGTHS = [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16, 18, 20, 21, 24, 25, 27, 28, 30, 32]
GRIDS = [tuple(np.roll((g, 2, 3), r)) for g in LENGTHS for r in range(3) if g > 3 or r == 0] + [(12, 7, 10), (4, 11, 3)]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
def test_axis_lengths(grid):
    torch = torch_cuda()
    mesh = (2, 3, 1) if sum(grid) < 20 else (3, 1, 2)
    spec = synth.GridSpec(mesh, 2, tuple(int(x) for x in grid), n_emb=3, seed=3)
    rho = synth.pair_densities_k(spec)
    C = synth.bloch_orbitals(synth.grid_orbitals(spec, complex_orbitals=True), mesh)
    d = dm.make_desc(mesh, 2, int(np.prod(grid)), 3, sym=B.DMET_SYM_NONE, eri_pack=B.DMET_PACK_FULL)
    rd = torch.from_numpy(np.ascontiguousarray(rho.transpose(0, 1, 4, 2, 3))).cuda()
    out = torch.empty(81, dtype=torch.complex128, device="cuda")
    plan = dm.dmet_emb_plan(d, stream=torch.cuda.current_stream().cuda_stream)
    try:
        dm.dmet_emb_eri_fftdf(plan, rd, [torch.from_numpy(C).cuda()], spec.grid, spec.lattice, [out])
        st, _ = dm.dmet_emb_status(plan, 0)
    finally:
        dm.dmet_emb_destroy(plan)
    assert st == B.DMET_OK
    ref = of.embedded_eri_fftdf(rho, C, mesh, spec.lattice, spec.grid).ravel()
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-12 * np.abs(ref).max()

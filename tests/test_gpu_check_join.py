"""The orbital checks run beside the transforms on a stream of the plan. A call that returns an error after it queued
them joins them to the caller's stream all the same: a capture of that stream ends without an unjoined fork, and what
follows on the stream (another C in the same buffer, the next call's statistics) waits for them."""
import numpy as np
import pytest

import oracle
import synth
import paper_1909_08596_gb300 as dm
from paper_1909_08596_gb300 import binding as B

from gpu_helpers import rel_fro, torch_cuda

pytestmark = pytest.mark.gpu
MESH, NAO, NAUX, N = (4, 1, 1), 40, 24, 32


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


@pytest.fixture()
def sharded(torch):
    """A tensor-core plan of the shard {0} on a stream of its own, its inputs, and a q outside the shard."""
    spec = synth.LatticeSpec(MESH, NAO, NAUX, N, 1, 0.6, 0.0, 81, "r")
    L, (C,), _ = synth.make_problem(spec)
    stream = torch.cuda.Stream()
    d = B.make_desc(MESH, NAO, NAUX, N, prec=B.DMET_PREC_BF16X3, q_range=(0, 1))
    Ld, Cd = torch.from_numpy(L).cuda(), torch.from_numpy(C).cuda()
    out = torch.empty((1, NAUX, N, N), dtype=torch.complex128, device="cuda")
    plan = dm.dmet_emb_plan(d, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    yield plan, stream, L, C, Ld, Cd, out
    dm.dmet_emb_destroy(plan)


def refused(plan, Ld, Cd, out):
    with pytest.raises(B.DmetError):
        dm.dmet_emb_transform_3idx(plan, 0, Ld, [Cd], 2, 3, [out])


def test_capture_ends_after_an_error_return(torch, sharded):
    plan, stream, L, C, Ld, Cd, out = sharded
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        g.capture_begin(capture_error_mode="thread_local")
        try:
            refused(plan, Ld, Cd, out)
        finally:
            g.capture_end()
        g.replay()
    stream.synchronize()


def test_next_call_after_an_error_return(torch, sharded):
    plan, stream, L, C, Ld, Cd, out = sharded
    good = Cd.clone()
    for _ in range(20):
        with torch.cuda.stream(stream):
            Cd.mul_(3.0)                     # not orthonormal: the refused call's checks must not reach the next one
            refused(plan, Ld, Cd, out)
            Cd.copy_(good)
            dm.dmet_emb_transform_3idx(plan, 0, Ld, [Cd], 0, 1, [out])
        st, stats = dm.dmet_emb_status(plan, 0)
        assert st == B.DMET_OK, stats
    ref = oracle.embedded_3idx(L, C, MESH)[0:1]
    assert rel_fro(out.cpu().numpy(), ref) < 2e-6

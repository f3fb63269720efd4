"""mraid_ccm for the correlation alone as a plan's first call (needs a GPU): on
shapes whose faster kernel needs a buffer for the sums it still works while the
stream is captured, and where that buffer cannot be had, with the same
correlations."""
import pytest

from gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub", [(19, 1, 1024, 600), (7, 3, 512, 800), (36, 64, 4096, 1)])
def test_first_call_without_a_buffer(n_beam, n_chan, n_s, n_sub):
    import torch
    m = lib()
    d = torch.randint(0, 256, (n_beam, n_sub * n_s, n_chan), dtype=torch.uint8, device="cuda")
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        assert m.mraid_gram_kernel(plan.handle, d) in ("gram_u8", "gram_tcl")
        want = plan.ccm(d, sums=False)[1]
        plan.sync()
    got = torch.zeros_like(want)
    stream = torch.cuda.Stream()
    with m.Plan(n_beam, n_chan, n_s, n_sub, stream=stream) as plan:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            m.mraid_ccm(plan.handle, d, None, got)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want)
    got.zero_()
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        m.mraid_inject_fault(plan.handle, m.FAULT_ALLOC)
        m.mraid_ccm(plan.handle, d, None, got)
        plan.sync()
        assert torch.equal(got, want)

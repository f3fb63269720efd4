"""The tuner times the eigensolvers with eigenvalues (needs a GPU): without
them variants 4 and 5 run one of their two kernels, a third of the time."""
import pytest

from gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam", [13, 19])
def test_eigensolver_times_include_the_eigenvalues(n_beam):
    import torch
    m = lib()
    n_chan, n_s, n_sub = 2048, 64, 64
    g = torch.Generator(device="cuda")
    g.manual_seed(n_beam)
    d = torch.randint(0, 256, (n_beam, n_sub * n_s, n_chan), dtype=torch.uint8, device="cuda", generator=g)
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        corr = plan.ccm(d, sums=False)[1]
        out = torch.empty(plan.n_cells, n_beam, device="cuda")
        stat = torch.empty(plan.n_cells, device="cuda")
        times = {}
        for evals in (None, out):
            for _ in range(3):
                m.mraid_eig(plan.handle, corr, evals, None, stat)
            runs = []
            for _ in range(9):
                e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                e0.record()
                for _ in range(4):
                    m.mraid_eig(plan.handle, corr, evals, None, stat)
                e1.record()
                torch.cuda.synchronize()
                runs.append(e0.elapsed_time(e1) / 4)
            times[evals is not None] = sorted(runs)[4]
        _, ms = m.mraid_autotune(plan.handle, d, 5)
    # between the two, nearer the one with eigenvalues
    middle = (times[True] * times[False]) ** 0.5
    assert times[True] > 1.5 * times[False]
    assert ms["e4"] > middle and ms["e5"] > middle, (ms, times)

"""The 8-bit Gram of narrow blocks (needs a GPU): its sums equal the CUDA-core
Gram's bit for bit wherever the rule by shape sends them, also where several
CTAs share an SM (more 32-channel items than SMs), and the rule's choice is
not the slower kernel by far."""
import pytest

from gpu_util import lib

pytestmark = pytest.mark.gpu


def block(n_beam, n_chan, n_s, n_sub, offset=0):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n_beam + n_chan)
    size = n_beam * n_sub * n_s * n_chan
    return torch.randint(0, 256, (size + offset,), dtype=torch.uint8, device="cuda", generator=g)[offset:]


@pytest.mark.parametrize("n_beam", [2, 7, 13, 19, 23])
@pytest.mark.parametrize("n_chan,n_s,n_sub,offset", [
    (1, 40, 1000, 0), (3, 100, 700, 0), (16, 64, 700, 0), (16, 2050, 170, 0),
    (17, 90, 400, 0), (24, 128, 330, 0), (28, 200, 310, 0), (20, 1030, 200, 4),
    (32, 100, 310, 3), (64, 16, 153, 0),
])
def test_same_sums_as_the_cuda_cores(n_beam, n_chan, n_s, n_sub, offset):
    import torch
    m = lib()
    d = block(n_beam, n_chan, n_s, n_sub, offset)
    got = {}
    for variant in (0, -1):
        with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
            m.mraid_set_variant(plan.handle, variant)
            sums, corr = plan.ccm(d)
            plan.sync()
            got[variant] = sums, corr
    assert torch.equal(got[0][0], got[-1][0])
    # float results of the same exact sums
    assert (got[0][1] - got[-1][1]).abs().max() <= 2e-6


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub", [
    (19, 1, 1024, 2000), (7, 8, 1024, 500), (36, 2, 512, 2000), (2, 17, 512, 1000),
    (13, 3, 64, 5000), (7, 40, 512, 400), (19, 16, 1024, 500),
])
def test_narrow_blocks_are_not_slower_than_the_cuda_cores(n_beam, n_chan, n_s, n_sub):
    import torch
    m = lib()
    d = block(n_beam, n_chan, n_s, n_sub)
    times = {}
    for variant in (0, -1):
        with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
            m.mraid_set_variant(plan.handle, variant)
            corr = torch.empty(plan.n_cells, n_beam * (n_beam + 1) // 2, device="cuda")
            runs = []
            for _ in range(9):
                e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                torch.cuda._sleep(100000)
                e0.record()
                for _ in range(3):
                    m.mraid_ccm(plan.handle, d, None, corr)
                e1.record()
                torch.cuda.synchronize()
                runs.append(e0.elapsed_time(e1) / 3)
            times[variant] = sorted(runs)[4]
    assert times[0] < 1.25 * times[-1], times

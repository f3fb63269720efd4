"""The plain copies of the 8-bit Gram from 24 beams on, where two groups of
threads (four for 8-byte copies) share a stage's beams (needs a GPU): beam
counts that leave the last group with more, fewer and no beams than the others,
for copies of 8, 4 and single bytes, and a block whose last channels have no
whole word. Sums equal to the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam", [24, 25, 33, 39])
@pytest.mark.parametrize("n_chan,offset", [(40, 0), (36, 0), (34, 0), (40, 3), (1, 0)])
@pytest.mark.parametrize("n_s", [40, 1030])
def test_every_beam_is_copied(n_beam, n_chan, offset, n_s):
    import torch
    m = lib()
    n_sub = 2
    rng = np.random.default_rng(n_beam * 100 + n_chan)
    data = rng.integers(0, 256, size=(n_beam, n_sub * n_s, n_chan), dtype=np.uint8)
    buf = torch.zeros(data.size + offset, dtype=torch.uint8, device="cuda")
    buf[offset:] = torch.from_numpy(data.reshape(-1)).cuda()
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        sums = plan.ccm(buf[offset:], corr=False)[0]
        plan.sync()
    iu = np.triu_indices(n_beam + 1)
    G = np.stack([oracle.cell_gram(data, n_s, k, c) for k in range(n_sub) for c in range(n_chan)])
    np.testing.assert_array_equal(sums.cpu().numpy(), G[:, iu[0], iu[1]])


def test_no_sample_is_copied_twice():
    """At odd addresses the copies bound the kernel, so a beam costs 36 beams
    about what it costs 23 (0.87 measured; 1.49 when every beam was copied by
    two groups)."""
    import torch
    m = lib()
    n_chan, n_s, n_sub = 1001, 1000, 20
    d = torch.randint(0, 256, (36 * n_sub * n_s * n_chan,), dtype=torch.uint8, device="cuda")
    per_beam = []
    for n_beam in (23, 36):
        with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
            corr = torch.empty(plan.n_cells, n_beam * (n_beam + 1) // 2, device="cuda")
            runs = []
            for _ in range(8):
                e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                torch.cuda._sleep(100000)
                e0.record()
                m.mraid_ccm(plan.handle, d, None, corr)
                e1.record()
                torch.cuda.synchronize()
                runs.append(e0.elapsed_time(e1))
            per_beam.append(sorted(runs[1:])[3] / n_beam)
    assert per_beam[1] < 1.2 * per_beam[0], per_beam

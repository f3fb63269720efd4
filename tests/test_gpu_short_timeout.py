"""An expired wait in a block of fewer stages than the copies' ring is deep
(needs a GPU): the kernel waits for the copies in flight alone, not for the
ring's other slots, so the call returns after one wait limit, not a dozen."""
import time

import numpy as np
import pytest

from gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam,stage", [(19, 0), (19, 1), (36, 0)])
def test_a_short_block_times_out_once(n_beam, stage):
    import torch
    m = lib()
    n_chan, n_s, n_sub, limit = 32, 32, 1, 0.2
    d = torch.from_numpy(np.random.default_rng(5).integers(
        0, 256, size=(n_beam, n_sub * n_s, n_chan), dtype=np.uint8)).cuda()
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        ref = plan.ccm(d, sums=False)[1].cpu()
        m.mraid_set_wait_limit(plan.handle, int(limit * 1e9))
        m.mraid_inject_fault(plan.handle, m.FAULT_WITHHOLD_STAGE, stage)
        t0 = time.monotonic()
        plan.ccm(d, sums=False)
        with pytest.raises(m.MraidError) as e:
            plan.sync()
        took = time.monotonic() - t0
        assert e.value.status == 5
        assert limit * 0.9 < took < 4 * limit, took
        corr = plan.ccm(d, sums=False)[1]
        plan.sync()
        assert torch.equal(corr.cpu(), ref)

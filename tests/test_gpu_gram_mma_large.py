"""The 8-bit Gram from register fragments where a warp holds four channels (24
to 39 beams) and where a sub-integration takes several 1024-sample pieces
(needs a GPU): beam counts around the 8-beam blocks, channel counts around the
work items, the last piece of one sample, of less than a step and of full
length, and sample buffers that no tensor map takes. The sums are integers:
equal to the oracle's bit for bit, and the correlation within the rounding of
its float result."""
import numpy as np
import pytest

import oracle
from gpu_util import CORR_TOL, lib, unpack_corr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub,offset", [
    (24, 48, 1024, 1, 0),    # four blocks; 32 + 16 channels
    (31, 32, 1056, 2, 0),    # full fourth block; two pieces
    (32, 20, 70, 2, 4),      # the row of ones opens the fifth block; 4-byte copies
    (36, 16, 15, 3, 0),      # less than a step
    (39, 33, 2050, 1, 0),    # full fifth block; three pieces, byte loads
    (27, 40, 100, 2, 1),     # misaligned buffer
    (7, 144, 1025, 2, 0),    # a piece and one sample; 128 + 16 channels
    (13, 128, 3072, 1, 0),   # three whole pieces
    (19, 80, 2047, 2, 0),    # half-filled last block
    (22, 72, 2048, 1, 8),    # 8-byte copies
    (5, 1000, 520, 5, 0),    # few beams by plain copies, more items than SMs
    (2, 24, 640, 2, 0),      # fewer: CUDA cores
    (9, 65, 40, 1, 3),       # odd addresses: word pairs, single bytes at both ends
])
def test_sums_exact(n_beam, n_chan, n_s, n_sub, offset):
    import torch
    m = lib()
    rng = np.random.default_rng(n_beam * 1000 + n_chan)
    data = rng.integers(0, 256, size=(n_beam, n_sub * n_s, n_chan), dtype=np.uint8)
    data[0] = 0                # saturated beams: products at the centring's extremes
    data[-1, :, ::2] = 255
    buf = torch.zeros(data.size + offset, dtype=torch.uint8, device="cuda")
    buf[offset:] = torch.from_numpy(data.reshape(-1)).cuda()
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        sums, corr = plan.ccm(buf[offset:])
        plan.sync()
    iu = np.triu_indices(n_beam + 1)
    G = np.stack([oracle.cell_gram(data, n_s, k, c) for k in range(n_sub) for c in range(n_chan)])
    np.testing.assert_array_equal(sums.cpu().numpy(), G[:, iu[0], iu[1]])
    r = np.stack([oracle.corr_from_gram(g)[0] for g in G])
    assert np.abs(unpack_corr(corr.cpu().numpy(), n_beam) - r).max() <= CORR_TOL

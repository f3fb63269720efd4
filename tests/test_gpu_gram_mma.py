"""The 8-bit Gram for up to 23 beams at the edges of its tiles (needs a GPU):
beam counts around the 8-beam blocks and the half-filled last block, channel
counts around the 32-, 64-, 96- and 128-channel work items, sample counts
around the 16-sample steps and the 1024-sample pieces, and sample buffers
that no tensor map takes (odd channel counts and byte offsets). The sums are
integers: equal to the oracle's bit for bit, and the correlation within the
rounding of its float result."""
import numpy as np
import pytest

import oracle
from gpu_util import CORR_TOL, lib, unpack_corr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub,offset", [
    (2, 16, 16, 2, 0),       # smallest: one block, one step
    (7, 144, 1024, 1, 0),    # full first block (with the row of ones), 128 + 16 channels
    (8, 64, 1040, 2, 0),     # the row of ones opens the second block; two pieces
    (15, 32, 33, 3, 0),      # full second block; two steps and one sample
    (16, 96, 15, 3, 0),      # less than a step
    (19, 112, 2049, 1, 0),   # half-filled last block; 96 + 16 channels; three pieces
    (20, 80, 48, 2, 0),      # full last block
    (23, 33, 100, 2, 0),     # odd channel count: byte loads
    (19, 100, 70, 2, 4),     # 4-byte copies
    (13, 72, 64, 2, 8),      # 8-byte copies
    (19, 64, 64, 2, 1),      # misaligned buffer
])
@pytest.mark.parametrize("variant", [0, 1])
def test_sums_exact_at_tile_edges(n_beam, n_chan, n_s, n_sub, offset, variant):
    import torch
    m = lib()
    rng = np.random.default_rng(n_beam * 1000 + n_chan)
    data = rng.integers(0, 256, size=(n_beam, n_sub * n_s, n_chan), dtype=np.uint8)
    data[0] = 0                # saturated beams: products at the centring's extremes
    data[-1, :, ::2] = 255
    buf = torch.zeros(data.size + offset, dtype=torch.uint8, device="cuda")
    buf[offset:] = torch.from_numpy(data.reshape(-1)).cuda()
    d = buf[offset:]
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        m.mraid_set_variant(plan.handle, variant)
        sums, corr = plan.ccm(d)
        plan.sync()
    M = n_beam + 1
    iu = np.triu_indices(M)
    G = np.stack([oracle.cell_gram(data, n_s, k, c) for k in range(n_sub) for c in range(n_chan)])
    np.testing.assert_array_equal(sums.cpu().numpy(), G[:, iu[0], iu[1]])
    r = np.stack([oracle.corr_from_gram(g)[0] for g in G])
    assert np.abs(unpack_corr(corr.cpu().numpy(), n_beam) - r).max() <= CORR_TOL

"""Masking at the sizes where the kernel changes (needs a GPU): one cell, part
of a quad, one CTA, the first cluster sizes, the last cell count that fits a
cluster and the first that does not, with preserved channels, buffers that
allow no vector access, and values the fit must survive (infinities, NaN)."""
import numpy as np
import pytest

import oracle
from gpu_util import lib

pytestmark = pytest.mark.gpu


def statistic(n, seed):
    rng = np.random.default_rng(seed)
    s = rng.normal(0.08, 0.004, n).astype(np.float32)
    hot = rng.random(n) < 0.05
    s[hot] = rng.uniform(0.1, 0.95, hot.sum()).astype(np.float32)
    return s, rng


@pytest.mark.parametrize("n_chan,n_sub,offset", [
    (1, 1, 0), (3, 1, 0), (17, 61, 1), (128, 128, 0), (16385, 1, 0), (1000, 33, 0), (131073, 1, 1),
    (54272, 16, 0),     # 16 CTAs of 53 x 1024 cells, full
    (868353, 1, 0),     # one cell more
])
@pytest.mark.parametrize("preserve", [False, True])
def test_mask_matches_oracle(n_chan, n_sub, offset, preserve):
    import torch
    m = lib()
    n = n_chan * n_sub
    s, rng = statistic(n, n)
    keep = None
    if preserve and n_chan > 8:
        keep = (rng.random(n_chan) < 0.1).astype(np.uint8)
    buf = torch.zeros(n + offset, device="cuda")
    buf[offset:] = torch.from_numpy(s).cuda()
    flags = torch.full((n + offset,), 7, dtype=torch.uint8, device="cuda")
    info = m.FlagInfo()
    with m.Plan(2, n_chan, 16, n_sub, keep=keep) as plan:
        m.mraid_flag(plan.handle, buf[offset:], flags[offset:], info)
        plan.sync()
    f_o, i_o = oracle.flag(s, n_chan, keep=keep)
    got = flags[offset:].cpu().numpy()
    # fits agree to FP32 rounding of the sums; cells that close to the
    # threshold may fall either way
    for k in ("mu", "sigma", "thresh"):
        assert abs(getattr(info, k) - i_o[k]) <= 1e-6 * max(abs(i_o[k]), 1e-12), k
    near = np.abs(s.astype(np.float64) - i_o["thresh"]) <= 1e-6 * i_o["thresh"]
    assert not np.any((got != f_o) & ~near)
    assert info.n_flagged == got.sum() and info.iterations == i_o["iterations"]
    if keep is not None:
        assert not np.any(got.reshape(n_sub, n_chan)[:, keep.astype(bool)])


@pytest.mark.parametrize("bad,flagged,fits,used", [
    (np.inf, 0, 1, 4096),        # infinite mean and threshold: nothing above it
    (np.nan, 0, 1, 4096),        # no threshold compares
    (-np.inf, 4095, 2, 1),       # threshold -inf: every other cell is above it
])
def test_infinities_and_nan(bad, flagged, fits, used):
    import torch
    m = lib()
    s, _ = statistic(4096, 3)
    s[100] = bad
    with m.Plan(2, 64, 16, 64) as plan:
        f, info = plan.flag(torch.from_numpy(s).cuda())
    assert int(f.sum()) == flagged and info["iterations"] == fits and info["converged"] == 1
    assert info["n_used"] == used

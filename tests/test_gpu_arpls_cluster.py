"""ArPLS where a cluster of CTAs shares a spectrum (needs a GPU): the first
length that takes two, lengths whose block rows leave a CTA with few or no
channels, and lengths that need four and eight CTAs' shared memory. Baselines
and solve counts against the oracle at the bandpass path's tolerance."""
import numpy as np
import pytest

import oracle
from gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1023, 1024, 1025, 2047, 2050, 4096, 4100, 8192, 9001, 20000])
@pytest.mark.parametrize("lam,itermax", [(1e5, 50), (10.0, 3)])
def test_long_spectra_match_oracle(n, lam, itermax):
    import torch
    m = lib()
    rng = np.random.default_rng(n)
    x = np.linspace(0, 1, n)
    y = 100 * (1 + 0.3 * np.sin(5 * x)) + rng.normal(0, 0.5, (3, n))
    y[:, rng.integers(0, n, n // 50)] += 20
    with m.Plan(2, 16, 16, 1) as plan:
        z, it = plan.arpls(torch.from_numpy(y).cuda(), lam=lam, ratio=1e-3, itermax=itermax)
    for i in range(3):
        zo, io = oracle.arpls(y[i], lam, 1e-3, itermax)
        assert int(it[i]) == io
        np.testing.assert_allclose(z[i].cpu().numpy(), zo, rtol=0, atol=1e-9 * np.abs(y[i]).max())

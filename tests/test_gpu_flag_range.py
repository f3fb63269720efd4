"""Masking of statistics of a large dynamic range (needs a GPU): finite
outliers far above everything else, a level far narrower than its distance
from zero, first cells unlike the rest or preserved, and equal cells, in one
CTA and over a cluster. Every one moves the mean away from the pivot that the
sums were taken about.

Tolerance: a cell's roundings (difference, square, sum of four) leave s2 / n an
error of 6 x 2^-24 at most, and the variance is taken where it is a tenth of
that or more: 3.6e-6 of the variance, 1.8e-6 of sigma, 5.4e-6 sigma in the
threshold at k = 3, and the mean's part below 1e-6 sigma."""
import numpy as np
import pytest

import oracle
from gpu_util import lib

pytestmark = pytest.mark.gpu


def level(n, mean, dev):
    return np.random.default_rng(n).normal(mean, dev, n).astype(np.float32)


def outlier(n, value, at):
    s = level(n, 0.08, 0.004)
    s[at] = value
    return s


def near_one(n):
    rng = np.random.default_rng(n)
    s = level(n, 0.0527, 5e-6)
    hot = rng.random(n) < 0.05
    s[hot] = rng.uniform(0.9, 1.0, hot.sum())
    return s


def hot_first(n):
    s = level(n, 0.08, 0.004)
    s[:1024] = np.random.default_rng(1).normal(0.9, 0.01, 1024)
    return s


@pytest.mark.parametrize("n,make,max_iter", [
    (4096, lambda n: outlier(n, 1e6, 3000), 64),
    (4096, lambda n: outlier(n, 1e5, 100), 64),
    (200000, lambda n: outlier(n, 1e6, 150000), 64),
    (200000, lambda n: outlier(n, 1e15, 7), 64),
    (16384, near_one, 64),
    (100000, near_one, 64),
    (4096, lambda n: level(n, 0.0527, 5e-6), 64),
    (4096, lambda n: level(n, 0.0527, 5e-8), 64),
    (16384, hot_first, 1),
    (50000, hot_first, 64),
    (5000, lambda n: np.full(n, 0.0527, np.float32), 64),
])
@pytest.mark.parametrize("first_preserved", [False, True])
def test_mask_of_a_large_range_matches_oracle(n, make, max_iter, first_preserved):
    import torch
    m = lib()
    s = make(n)
    keep = None
    if first_preserved:
        keep = np.zeros(n, np.uint8)
        keep[:1100] = 1
    with m.Plan(2, n, 16, 1, keep=keep, max_clip_iter=max_iter) as plan:
        f, info = plan.flag(torch.from_numpy(s).cuda())
    f_o, i_o = oracle.flag(s, n, keep=keep, max_iter=max_iter)
    tol = 1e-5 * i_o["sigma"] + 1e-12 * abs(i_o["mu"])  # and the oracle's own FP64 sums
    for k in ("mu", "sigma", "thresh"):
        assert abs(info[k] - i_o[k]) <= tol, (k, info[k], i_o[k])
    close = np.abs(s.astype(np.float64) - i_o["thresh"]) <= tol
    got = f.cpu().numpy()
    assert not np.any((got != f_o) & ~close), (int(got.sum()), int(f_o.sum()))
    assert info["n_flagged"] == got.sum() and info["iterations"] == i_o["iterations"]

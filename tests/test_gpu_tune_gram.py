"""Gram ids of the tuner (needs a GPU): every different launch is timed once
and reported for its aliases, and only an id with a launch of its own is
chosen."""
import pytest

from gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub,own", [
    (13, 1024, 256, 64, (-1, 0, 1)),    # 128-channel items, or 64
    (23, 4096, 64, 40, (-1, 0)),        # 64 is the shape's own choice
    (19, 64, 2048, 4, (-1, 0)),         # several pieces: one form
    (36, 64, 256, 4, (-1, 0)),          # 32 channels always
    (2, 1000, 1024, 2, (0,)),           # few beams by plain copies: CUDA cores by the rule
])
def test_only_different_launches_are_timed(n_beam, n_chan, n_s, n_sub, own):
    import torch
    m = lib()
    d = torch.randint(0, 256, (n_beam, n_sub * n_s, n_chan), dtype=torch.uint8, device="cuda")
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        (gram, _), ms = m.mraid_autotune(plan.handle, d, 3)
    assert gram in own, (gram, ms)
    assert all(ms[f"g{v}"] == ms["g0"] for v in range(2, 10)), ms
    assert (ms["g1"] == ms["g0"]) == (1 not in own), ms
    if own == (0,):
        assert ms["g0"] == ms["g-1"], ms

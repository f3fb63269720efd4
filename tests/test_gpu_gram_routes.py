"""Which kernel forms the Gram (needs a GPU): mraid_gram_kernel names it by
shape, layout and variant, and every tensor-core kernel is tested as itself:
an expired wait is reported and leaves the plan usable (nothing faults or hangs
the device), a block with more work items than SMs on gram_tcl, and the
timescales on the CUDA-core Gram."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import lib

pytestmark = pytest.mark.gpu
TIMEOUT = 5


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub,offset,variant,bits,name", [
    (19, 4096, 1024, 2, 0, 0, 8, "gram_mma"),
    (19, 4096, 1024, 2, 0, 1, 8, "gram_mma"),
    (19, 4096, 1024, 2, 0, -1, 8, "gram_u8"),
    (19, 4096, 1024, 2, 1, 0, 8, "gram_mma, plain copies"),
    (19, 1001, 1000, 4, 0, 0, 8, "gram_mma, plain copies"),
    (19, 1, 1024, 2000, 0, 0, 8, "gram_u8"),       # narrow: CUDA cores by the rule
    (36, 2048, 1024, 2, 0, 0, 8, "gram_mma"),
    (36, 64, 4096, 1, 0, 0, 8, "gram_tcl"),        # few long sub-integrations
    (64, 256, 512, 4, 0, 0, 8, "gram_tcl"),
    (64, 100, 512, 4, 0, 0, 8, "gram_u8"),
    (19, 64, 128, 4, 0, 0, 32, "gram_tc_f32"),
    (19, 64, 128, 4, 0, -1, 32, "gram_f32"),
])
def test_names(n_beam, n_chan, n_s, n_sub, offset, variant, bits, name):
    import torch
    m = lib()
    at = torch.empty(64, dtype=torch.uint8, device="cuda")[offset:]
    with m.Plan(n_beam, n_chan, n_s, n_sub, bit_depth=bits) as plan:
        m.mraid_set_variant(plan.handle, variant)
        assert m.mraid_gram_kernel(plan.handle, at) == name


def test_no_plan():
    assert lib().mraid_gram_kernel(None, None) == ""


@pytest.mark.parametrize("n_beam,n_chan,n_s,n_sub,pol2,name", [
    (64, 32, 2048, 2, False, "gram_tcl"),
    (36, 64, 4096, 1, False, "gram_tcl"),
    (36, 64, 512, 4, False, "gram_mma"),
    (19, 33, 1024, 4, False, "gram_mma, plain copies"),
    (36, 40, 512, 4, False, "gram_mma, plain copies"),
    (19, 32, 1024, 4, True, None),
])
def test_an_expired_wait_is_reported_and_the_plan_recovers(n_beam, n_chan, n_s, n_sub, pol2, name):
    import torch
    m = lib()
    rng = np.random.default_rng(n_beam)
    shape = (n_beam * (2 if pol2 else 1), n_sub * n_s, n_chan)
    d = torch.from_numpy(rng.integers(0, 256, size=shape, dtype=np.uint8)).cuda()
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        if name:
            assert m.mraid_gram_kernel(plan.handle, d) == name
        call = plan.ccm_pol2 if pol2 else plan.ccm
        m.mraid_profile_enable(plan.handle)
        ref = call(d)
        plan.sync()
        assert not pol2 or "pol2_fold" not in m.mraid_profile_read(plan.handle)
        m.mraid_set_wait_limit(plan.handle, 50_000_000)
        for stage in (0, 5):
            m.mraid_inject_fault(plan.handle, m.FAULT_WITHHOLD_STAGE, stage)
            call(d)
            with pytest.raises(m.MraidError) as e:
                plan.sync()
            assert e.value.status == TIMEOUT, e.value
            got = call(d)
            plan.sync()
            assert all(torch.equal(a, b) for a, b in zip(got, ref)), stage


def test_gram_tcl_with_more_items_than_sms():
    import torch
    m = lib()
    n_beam, n_chan, n_s, n_sub = 64, 256, 512, 12    # 192 boxes of 16 channels, more than one pass each
    rng = np.random.default_rng(5)
    data = np.clip(np.rint(rng.normal(128, 20, size=(n_beam, n_sub * n_s, n_chan))), 0, 255).astype(np.uint8)
    d = torch.from_numpy(data).cuda()
    with m.Plan(n_beam, n_chan, n_s, n_sub) as plan:
        assert m.mraid_gram_kernel(plan.handle, d) == "gram_tcl"
        sums = plan.ccm(d, corr=False)[0]
        m.mraid_set_variant(plan.handle, -1)
        sums2 = plan.ccm(d, corr=False)[0]
        plan.sync()
    assert torch.equal(sums, sums2)
    got, iu = sums.cpu().numpy(), np.triu_indices(n_beam + 1)
    for cell in rng.choice(n_sub * n_chan, size=16, replace=False):
        k, c = divmod(int(cell), n_chan)
        assert np.array_equal(got[cell], oracle.cell_gram(data, n_s, k, c)[iu]), cell


def test_timescales_on_the_cuda_core_gram():
    import torch
    m = lib()
    nb, nc, ns, nk = 13, 40, 64, 12
    cfg = synth.SMALL.replace(n_beam=nb, n_chan=nc, n_samp_sub=ns, n_sub=nk, n_burst=1)
    d = torch.from_numpy(synth.generate(cfg)).cuda()
    with m.Plan(nb, nc, ns, nk) as plan:
        m.mraid_set_variant(plan.handle, -1)
        assert m.mraid_gram_kernel(plan.handle, d) == "gram_u8"
        levels = plan.multires(d, [1, 2, 3, nk])
    for lv in levels:
        f = lv["factor"]
        with m.Plan(nb, nc, f * ns, nk // f, beam_stride=nk * ns * nc) as p2:
            out = p2.run(d, evals=False, q1=False)
        assert torch.equal(lv["stat"], out["stat"]) and torch.equal(lv["flags"], out["flags"])

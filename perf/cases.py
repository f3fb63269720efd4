"""Performance cases of the eigenvalue RFI flagger.

A case is one call of a public entry point on a block that is already in
device memory, as an observing program makes it: the whole path (`Plan.run`),
its two-polarisation, several-timescale and bandpass forms, the correlation
alone, or the decomposition alone. Shapes follow the FAST 19-beam receiver
(4096 channels, 1024-sample sub-integrations), the 13-, 36- and 72-beam
receivers of the batched form, the small test block, and blocks that fit no
tile (odd channel and sample counts).
"""
import concurrent.futures
import math

import numpy as np
import torch

import paper_2512_16278_gb300 as m

# Sub-interval lengths of Table 1 (0.05 s to 10 s) in 1024-sample
# sub-integrations of 49.152 us.
TABLE1 = (1, 4, 10, 20, 40, 100, 200)


def _case(form, beams, chans, samples, subs, bits=8, evals=False, q1=False, refine=False):
    return {"form": form, "beams": beams, "chans": chans, "samples": samples, "subs": subs,
            "bits": bits, "evals": evals, "q1": q1, "refine": refine}


def listed():
    return [
        # a quick look at a few channels of a live stream: latency and launches
        dict(_case("run", 19, 128, 256, 8), name="quicklook"),
        # the small test block, every output: 16 384 short cells
        dict(_case("run", 19, 64, 128, 256, evals=True, q1=True), name="small_block"),
        # a live 0.2 s of the FAST receiver, with the beams that each flagged
        # cell affects
        dict(_case("run", 19, 4096, 1024, 4, evals=True, q1=True, refine=True), name="fast_live"),
        # the FAST block, 10 s, every output: what an archive run does
        dict(_case("run", 19, 4096, 1024, 200, evals=True, q1=True), name="fast_block"),
        # 5 s of the 13-, 36- and 72-beam receivers, masks and eigenvalues
        dict(_case("run", 13, 1024, 512, 152, evals=True), name="rx13"),
        dict(_case("run", 36, 2048, 2048, 38, evals=True), name="rx36"),
        dict(_case("run", 72, 1024, 4096, 19, evals=True), name="rx72"),
        # sizes that fit no tile: 1000 channels (a cut band), 1000 samples
        # (a rounded sub-integration time)
        dict(_case("run", 19, 1000, 1000, 40, evals=True), name="ragged"),
        # both recorded polarisations, 2 s
        dict(_case("pol2", 19, 4096, 1024, 40), name="two_polarisations"),
        # float32 beamformer output, 1 s: the correlation
        dict(_case("ccm", 19, 4096, 1024, 20, bits=32), name="float32"),
        # Table 1's seven timescales over 10 s of a quarter of the band
        dict(_case("multires", 19, 1024, 1024, 200), name="timescales"),
        # the bandpass-centred reading over 2 s, 1 s fit intervals
        dict(_case("bandpass", 19, 4096, 1024, 40, evals=True), name="bandpass"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["run"] * 6 + ["pol2", "pol2", "ccm", "ccm", "multires", "bandpass", "eig"])
    bits = 32 if form == "ccm" and rng.random() < 0.6 else 8
    # receivers: mostly up to 23 beams, phased-array feeds up to 90
    beams = rng.randint(4, 23) if rng.random() < 0.6 or form != "run" else rng.randint(24, 90)
    chans, samples = _log(rng, 32, 4096), _log(rng, 64, 4096)
    if rng.random() < 0.7:  # whole tiles, as receivers deliver them
        chans = max(16, chans // 16 * 16)
        samples = max(64, samples // 64 * 64)
    if bits == 32:
        samples = min(samples, 1024)
    # block sizes over the whole range: 1 MB to 3 GB of samples, at most
    # 200 000 cells
    sample_bytes = beams * chans * samples * (4 if bits == 32 else 1) * (2 if form == "pol2" else 1)
    subs = max(1, _log(rng, 1e6, 3e9) // sample_bytes)
    subs = min(subs, 200, max(1, 200000 // chans))
    evals = form in ("run", "pol2", "bandpass", "eig") and rng.random() < 0.6
    q1 = form in ("run", "eig") and beams <= 23 and samples >= 256 and rng.random() < 0.4
    return _case(form, beams, chans, samples, subs, bits=bits, evals=evals, q1=q1)


def _factors(c):
    return [f for f in TABLE1 if f <= c["subs"]]


def _block(c, seed):
    """The block's samples [beam][time][chan]: noise of 20 counts around 128
    times a bandpass gain per beam and channel; 2 % of the channels carry a
    tone and 1 % of the sub-integrations a burst in every beam, 0.1 % of the
    cells a pulse in one beam."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    B, C, S, K = c["beams"], c["chans"], c["samples"], c["subs"]
    blocks = B * (2 if c["form"] == "pol2" else 1)
    rng = np.random.default_rng(seed)
    gain = torch.from_numpy(rng.uniform(0.7, 1.3, (blocks, 1, C)).astype(np.float32)).cuda()
    amp = torch.from_numpy(rng.uniform(0.5, 1.5, (blocks, 1, 1)).astype(np.float32)).cuda()
    tone = np.zeros(C, np.float32)
    tone[rng.permutation(C)[:max(1, round(0.02 * C))]] = 15.0
    tone = torch.from_numpy(tone).cuda()
    wave = torch.sin(torch.arange(S, device="cuda", dtype=torch.float32) * (2 * math.pi / 16))
    burst = set(rng.permutation(K)[:max(1, round(0.01 * K))].tolist()) if K > 1 else set()
    spikes = max(1, round(0.001 * C * K))
    where = {}
    for b, ch, k, t in zip(rng.integers(0, blocks, spikes), rng.integers(0, C, spikes),
                           rng.integers(0, K, spikes), rng.integers(0, max(1, S - 16), spikes)):
        where.setdefault(int(k), []).append((int(b), int(ch), int(t)))
    out = torch.empty(blocks, K * S, C, device="cuda",
                      dtype=torch.uint8 if c["bits"] == 8 else torch.float32)
    for k in range(K):
        x = torch.randn(blocks, S, C, device="cuda", generator=g)
        x.mul_(20.0).add_(128.0).mul_(gain)
        x.add_(amp * (tone[None, None, :] * wave[None, :, None]))
        if k in burst:
            x[:, S // 3: S // 3 + max(1, S // 2)] += 40.0 * amp
        if k in where:
            b, ch, t = (torch.tensor(v, device="cuda") for v in zip(*where[k]))
            tt = (t[:, None] + torch.arange(16, device="cuda")).clamp_(max=S - 1)
            x.index_put_((b[:, None], tt, ch[:, None]),
                         torch.full(tt.shape, 80.0, device="cuda"), accumulate=True)
        if c["bits"] == 8:
            x.round_().clamp_(0, 255)
        out[:, k * S:(k + 1) * S] = x
    return out


def prepare(case, seed):
    data = _block(case, seed)
    plan = m.Plan(case["beams"], case["chans"], case["samples"], case["subs"],
                  bit_depth=case["bits"])
    if case["form"] == "eig":  # the correlations, as the first step of the path left them
        data = plan.ccm(data, sums=False)[1]
    return {"case": case, "plan": plan, "data": data}


_MASK = ("mu", "sigma", "thresh")


def _report(info):
    return [float(info[k]) for k in _MASK]


def run(state):
    c, plan, data = state["case"], state["plan"], state["data"]
    if c["form"] == "ccm":
        sums, corr = plan.ccm(data, sums=c["bits"] == 8)
        return {"sums": sums, "corr": corr}
    if c["form"] == "eig":
        evals, q1, stat = plan.eig(data, evals=c["evals"], q1=c["q1"])
        return {"evals": evals, "q1": q1, "stat": stat}
    if c["form"] == "multires":
        return [{"stat": l["stat"], "flags": l["flags"], "mask": _report(l["info"])}
                for l in plan.multires(data, _factors(c))]
    if c["form"] == "pol2":
        out = plan.run_pol2(data, evals=c["evals"], q1=False)
    elif c["form"] == "bandpass":
        out = plan.run_bandpass(data, evals=c["evals"])
    else:
        out = plan.run(data, evals=c["evals"], q1=c["q1"])
    res = {k: out[k] for k in ("evals", "q1", "stat", "flags", "bandpass") if out.get(k) is not None}
    res["mask"] = _report(out["info"])
    if c["refine"]:
        res["bits"], res["mu_sigma"] = plan.refine(out["q1"], out["flags"])
    return res


def work(case):
    """Samples read once, results written once; the upper triangle of every
    cell's products, and the dense reduction of its matrix."""
    B, C, S, K = case["beams"], case["chans"], case["samples"], case["subs"]
    cells, pairs = C * K, B * (B + 1) // 2
    nbytes = cells * B * S * (case["bits"] // 8) * (2 if case["form"] == "pol2" else 1)
    flops = 2 * cells * pairs * S
    dense = 4 * B ** 3 // 3
    if case["form"] == "ccm":
        nbytes += cells * pairs * 4 + (cells * (B + 1) * (B + 2) * 4 if case["bits"] == 8 else 0)
        return {"bytes": nbytes, "flops": flops}
    out = (4 * B if case["evals"] else 0) + (4 * B if case["q1"] else 0)
    if case["form"] == "eig":
        return {"bytes": cells * (pairs * 4 + 4 + out), "flops": cells * dense}
    if case["form"] == "multires":
        cells = sum(K // f for f in _factors(case)) * C
    nbytes += cells * (5 + out)
    if case["form"] == "bandpass":
        nbytes += -(-K // 20) * B * C * 4
    if case["refine"]:
        nbytes += cells * (4 * B + 1 + 4 * ((B + 31) // 32))
    return {"bytes": nbytes, "flops": flops + cells * dense}


# ---------------------------------------------------------------- 64 bits

def _sums(c, data):
    """Per cell the raw second moments [cell][B][B] and sums [cell][B] (64-bit)."""
    B, C, S, K = c["beams"], c["chans"], c["samples"], c["subs"]
    g2 = torch.empty(K * C, B, B, dtype=torch.float64, device="cuda")
    g1 = torch.empty(K * C, B, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // (B * S))
    for k in range(K):
        for c0 in range(0, C, step):
            x = data[:, k * S:(k + 1) * S, c0:c0 + step].double()
            if c["form"] == "pol2":
                x = x[:B] + x[B:]
            x = x.permute(2, 0, 1).contiguous()
            at = slice(k * C + c0, k * C + c0 + x.shape[0])
            if c["bits"] == 32:  # about the cell's mean: no cancellation
                x = x - x.mean(2, keepdim=True)
            g1[at] = x.sum(2)
            torch.bmm(x, x.transpose(1, 2), out=g2[at])
    return g2, g1


def _corr(g2, g1, n):
    cov = n * g2 - g1[:, :, None] * g1[:, None, :]
    sd = torch.diagonal(cov, dim1=1, dim2=2).clamp(min=0).sqrt()
    inv = torch.where(sd > 0, 1 / sd, torch.zeros_like(sd))
    r = cov * inv[:, :, None] * inv[:, None, :]
    torch.diagonal(r, dim1=1, dim2=2).fill_(1.0)
    return r


def _eig(r, vectors):
    """Eigenvalues (largest first), dominant eigenvector and statistic."""
    a = r.cpu().numpy()
    step = max(1, 4000000 // a.shape[1] ** 3 + 16)
    parts = [a[i:i + step] for i in range(0, a.shape[0], step)]
    with concurrent.futures.ThreadPoolExecutor(16) as pool:
        got = list(pool.map(np.linalg.eigh if vectors else np.linalg.eigvalsh, parts))
    ev = np.concatenate([g[0] if vectors else g for g in got])[:, ::-1]
    q1 = None
    if vectors:
        q1 = np.concatenate([g[1][:, :, -1] for g in got])
        big = np.take_along_axis(q1, np.abs(q1).argmax(1)[:, None], 1)
        q1 = torch.from_numpy(q1 * np.where(big < 0, -1.0, 1.0))
    stat = ev[:, 0] ** 2 / (ev ** 2).sum(1)
    return torch.from_numpy(ev.copy()), q1, torch.from_numpy(stat)


def _mask(stat, k=3.0):
    """[mean, deviation, threshold] of the converged Gaussian fit."""
    s = stat.numpy()
    used = np.ones(s.shape, bool)
    mu = sd = th = 0.0
    for _ in range(64):
        mu, sd = s[used].mean(), s[used].std()
        th = mu + k * sd
        new = used & ~(s > th)
        if new.sum() == used.sum():
            break
        used = new
    return [float(mu), float(sd), float(th)]


def exact(case, seed):
    c = case
    B, C, S, K = c["beams"], c["chans"], c["samples"], c["subs"]
    if c["form"] == "bandpass":  # the fit's stopping rule is the method's own
        return None
    if c["beams"] ** 3 * C * K > 2e10:
        return None
    g2, g1 = _sums(c, _block(c, seed))
    if c["form"] == "multires":
        res = []
        for f in _factors(c):
            n = K // f
            a2 = g2[:n * f * C].view(n, f, C, B, B).sum(1).view(-1, B, B)
            a1 = g1[:n * f * C].view(n, f, C, B).sum(1).view(-1, B)
            stat = _eig(_corr(a2, a1, f * S), False)[2]
            res.append({"stat": stat, "flags": None, "mask": _mask(stat)})
        return res
    r = _corr(g2, g1, S)
    if c["form"] == "ccm":
        i, j = torch.triu_indices(B, B, device="cuda")
        return {"sums": None, "corr": r[:, i, j]}
    ev, q1, stat = _eig(r, c["q1"])
    if c["form"] == "eig":
        return {"evals": ev if c["evals"] else None, "q1": q1, "stat": stat}
    res = {"stat": stat, "flags": None, "mask": _mask(stat)}
    if c["evals"]:
        res["evals"] = ev
    if c["q1"]:
        res["q1"] = q1
    if c["refine"]:
        res["bits"] = res["mu_sigma"] = None
    return res

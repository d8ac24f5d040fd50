"""The work that a user of this library has it do, as a list of measured cases.

Every case goes through the public entry points of ``paper_2512_00398_gb300``:
``hp_search`` (a whole single-pulse search of one filterbank), its stages
``hp_dedisperse`` and ``hp_detect`` + ``hp_merge`` on their own, ``Batch`` (many
files in one launch sequence) and ``Stream`` (beams pushed gulp by gulp).  Shapes
are those of ``workloads.py`` and of the tests: bands of 100 to 4096 channels over
1000-1500 MHz (or the tiny band's 250 MHz), 48 or 64 us sampling, Gaussian noise
with dispersed pulses, and for the stress recipe broadband spikes, tones and a
baseline drift.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2512_00398_gb300 as hp
from paper_2512_00398_gb300 import synth, workloads

K_DM = 4148.808
CAND_CAPACITY = 1 << 16
GULP_CANDS = 256            # candidates kept per streamed gulp


# ------------------------------------------------------------------ the cases
def _search(name, nchans, nsamps, ndm, dm_hi, wmax, band=500.0, tsamp_us=49.152, grid="smearing",
            npulses=10, baseline="median", variant="plain", rfi=False, stress=False,
            raw_capacity=1 << 22, kind="search"):
    return {"name": name, "kind": kind, "nchans": nchans, "nsamps": nsamps, "ndm": ndm,
            "dm_hi": dm_hi, "wmax": wmax, "band": band, "tsamp_us": tsamp_us, "grid": grid,
            "npulses": npulses, "baseline": baseline, "variant": variant, "rfi": rfi,
            "stress": stress, "raw_capacity": raw_capacity}


def listed():
    return [
        # the smallest configuration: 2 s of a 128-channel band, 100 uniform trials;
        # what a quick-look monitor searches, bound by launches and latency
        _search("search tiny", 128, 32768, 100, 400.0, 64, band=250.0, tsamp_us=64.0,
                grid="uniform", npulses=3),
        # a short ragged recording (odd channel and sample counts, no alignment
        # anywhere) with the moving-mean baseline
        _search("search ragged mean", 1003, 50021, 201, 300.0, 512, tsamp_us=64.0,
                baseline="mean", npulses=3),
        # one gulp plus its overlap tail of the 4096-channel band: the unit of work of
        # a chunked search of a long observation
        _search("search gulp 4096ch", 4096, 163147, 1500, 2000.0, 4096, npulses=3),
        # a file of the multi-file workload: 2048 channels, 64 us, DM 0-1000
        _search("search 2048ch", 2048, 1 << 18, 750, 1000.0, 4096, tsamp_us=64.0, npulses=5),
        # the single-file flagship: 51.5 s of 4096 channels, 1500 trials on DM 0-2000
        _search("search fast", 4096, 1 << 20, 1500, 2000.0, 4096, npulses=20),
        # the stress recipe (spikes, tones, drift, DM 0-5000, 4000 trials) with RFI
        # mitigation on, half its full length
        _search("search stress rfi", 4096, 1 << 20, 4000, 5000.0, 8192, npulses=25, rfi=True,
                stress=True, raw_capacity=1 << 26),
        # the two-stage sub-band variant on the gulp's band, a longer chunk
        _search("search subband", 4096, 1 << 18, 1500, 2000.0, 4096, variant="subband", npulses=5),
        # per-width sigmas, as Heimdall normalises
        _search("search width sigma", 1024, 1 << 18, 750, 1000.0, 4096, variant="width_sigma",
                npulses=5),
        # dedispersed series alone (for a caller's own detection), odd lengths
        _search("dedisperse 1024ch", 1024, 200003, 400, 600.0, 64, tsamp_us=64.0, npulses=3,
                kind="dedisperse"),
        # detection and merging of a caller's dedispersed series
        _search("detect merge", 1, 300001, 700, 0.0, 4096, kind="detect", npulses=30),
        # eight files of uneven length, channel count and sampling time in one batch
        {"name": "batch 8 files", "kind": "batch", "nfiles": 8, "seed0": 100, "len_lo": 1 << 17,
         "len_hi": 1 << 19, "dm_hi": 1000.0, "wmax": 4096},
        # four beams of the 4096-channel band in steady state, four gulps each per pass,
        # from pinned host memory to candidates in host memory
        {"name": "stream 4 beams", "kind": "stream", "nbeams": 4, "ngulps": 4, "gulp": 8192,
         "nchans": 4096, "tsamp_us": 49.152, "ndm": 375, "dm_hi": 500.0, "wmax": 1024},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["search", "search", "search", "search", "dedisperse", "detect", "batch",
                       "stream"])
    if kind == "batch":
        return {"kind": "batch", "nfiles": rng.randint(2, 10), "seed0": rng.randint(0, 100000),
                "len_lo": 1 << 17, "len_hi": 1 << rng.randint(17, 19),
                "dm_hi": rng.uniform(300.0, 1000.0), "wmax": 1 << rng.randint(9, 12)}
    if kind == "stream":
        wmax = 1 << rng.randint(6, 10)
        nchans = _logint(rng, 128, 4096)
        dm_hi = rng.uniform(100.0, 500.0)
        tsamp = rng.choice([49.152, 64.0])
        # the gulps of a pass cover the tail (delay of the highest trial + widest boxcar),
        # so every pass searches the same beams' steady state
        tail = _max_delay(nchans, 500.0, tsamp, dm_hi) + wmax
        ngulps = rng.randint(2, 5)
        return {"kind": "stream", "nbeams": rng.randint(1, 6), "ngulps": ngulps,
                "gulp": max(2048, tail // ngulps + rng.randint(1, 3000)), "nchans": nchans,
                "tsamp_us": tsamp, "ndm": rng.randint(50, 400), "dm_hi": dm_hi, "wmax": wmax}
    if kind == "detect":
        return _drawn(_search("", 1, _logint(rng, 20000, 600000), _logint(rng, 20, 1500), 0.0,
                              1 << rng.randint(5, 12), kind="detect", npulses=rng.randint(1, 30),
                              baseline=rng.choice(["median", "median", "mean"])))
    nchans = rng.choice([_logint(rng, 100, 4096), _logint(rng, 100, 4096), 1024, 2048, 4096])
    wmax = 1 << rng.randint(6, 13 if kind == "search" else 7)
    tsamp = rng.choice([49.152, 64.0])
    dm_hi = math.exp(rng.uniform(math.log(150.0), math.log(2500.0)))
    maxd = _max_delay(nchans, 500.0, tsamp, dm_hi)
    nout = _logint(rng, max(8192, 2 * wmax), 1 << 20)
    nsamps = maxd + nout
    ndm = rng.randint(max(20, int(0.4 * dm_hi)), max(100, int(0.8 * dm_hi)))
    variant = "plain"
    if kind == "search":
        variant = rng.choice(["plain", "plain", "plain", "plain", "subband", "width_sigma", "decimate"])
    # at most the largest listed case's sums, and 2^30 (trial, sample) pairs
    while nout > 8192 and (nout * ndm * nchans > 1 << 43 or nout * ndm > 1 << 30):
        nout = nout * 3 // 4
        nsamps = maxd + nout
    if nsamps <= maxd + 2 * wmax:
        wmax = 64
    stress = kind == "search" and variant == "plain" and rng.random() < 0.25
    return _drawn(_search("", nchans, nsamps, ndm, dm_hi, wmax, tsamp_us=tsamp,
                          npulses=rng.randint(0, 12),
                          baseline=rng.choice(["median", "median", "median", "mean"]),
                          variant=variant, rfi=stress, stress=stress,
                          raw_capacity=1 << 26 if stress else 1 << 22, kind=kind))


def _drawn(case):
    return {k: v for k, v in case.items() if k != "name"}


# ------------------------------------------------------------------ the inputs
def _obs(case):
    nch = case["nchans"]
    return synth.Observation(nchans=nch, f_top=1500.0, chan_bw=-case.get("band", 500.0) / nch,
                             tsamp=case["tsamp_us"] * 1e-6, nsamps=case.get("nsamps", 0),
                             mean=128.0, sigma=16.0 if nch == 128 else 12.0)


def _max_delay(nchans, band, tsamp_us, dm):
    f_lo = 1500.0 - band * (nchans - 1) / nchans
    return int(math.ceil(K_DM * dm * (f_lo ** -2 - 1500.0 ** -2) / (tsamp_us * 1e-6)))


def _dm_list(case, obs):
    if case.get("grid") == "uniform":
        return synth.dm_list_uniform(0.0, case["dm_hi"], case["ndm"])
    return synth.dm_list_smearing(obs, 0.0, case["dm_hi"], case["ndm"])


def _pulses(obs, rng, n, dm_hi, t_hi):
    """Pulses of nominal S/N 8-30, FWHM 0.1-20 ms, arrival times inside the series."""
    out = []
    for _ in range(n):
        fwhm = math.exp(rng.uniform(math.log(0.1e-3), math.log(20e-3)))
        snr = rng.uniform(8.0, 30.0)
        amp = synth.amp_for_matched_snr(snr, fwhm / obs.tsamp, obs.nchans, obs.sigma)
        out.append((rng.uniform(0.0, dm_hi), rng.uniform(0.05, 0.95) * t_hi, fwhm, amp))
    return out


def _filterbank(obs, seed, pulses=(), stress=False):
    """uint8 [nsamps][nchans] on the GPU: radiometer noise, dispersed pulses and, for
    the stress recipe, spikes once per second, 5% of channels with tones and a drift."""
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 17)
    n, nch = obs.nsamps, obs.nchans
    f = obs.f_top + np.arange(nch) * obs.chan_bw
    x = torch.empty((n, nch), dtype=torch.uint8, device=dev)
    rows = max(256, (1 << 25) // nch)
    tone = None
    if stress:
        tone = torch.zeros(nch, device=dev)
        tone[torch.randperm(nch, generator=gen, device=dev)[: max(1, nch // 20)]] = 40.0
    arrivals = [(t0 + K_DM * dm * (f ** -2 - obs.f_top ** -2), fwhm, amp)
                for dm, t0, fwhm, amp in pulses]
    buf = torch.empty(min(rows, n) * nch, device=dev)
    for r0 in range(0, n, rows):
        r1 = min(n, r0 + rows)
        v = buf[: (r1 - r0) * nch].view(r1 - r0, nch)
        v.normal_(obs.mean, obs.sigma, generator=gen)
        for tau, fwhm, amp in arrivals:
            lo, hi = r0 * obs.tsamp - 4 * fwhm, r1 * obs.tsamp + 4 * fwhm
            a, b = np.searchsorted(tau, [lo, hi])      # channels that it crosses in this chunk
            if b <= a:
                continue
            i0 = max(r0, int((tau[a] - 4 * fwhm) / obs.tsamp))
            i1 = min(r1, int((tau[b - 1] + 4 * fwhm) / obs.tsamp) + 1)
            if i1 <= i0:
                continue
            t = torch.arange(i0, i1, device=dev, dtype=torch.float64) * obs.tsamp
            dt = ((t[:, None] - torch.from_numpy(tau[a:b]).to(dev)[None, :]) / fwhm).float()
            v[i0 - r0:i1 - r0, a:b] += amp * torch.exp(-4.0 * math.log(2.0) * dt * dt)
        if stress:
            t = torch.arange(r0, r1, device=dev, dtype=torch.float64) * obs.tsamp
            v += (10.0 * torch.sin(2.0 * math.pi * t / 10.0)).float()[:, None]
            v += tone[None, :]
            every = max(1, int(round(1.0 / obs.tsamp)))
            first = (every // 2 - r0) % every
            v[first::every] += 3.0 * obs.sigma
        x[r0:r1] = v.round_().clamp_(0.0, 255.0).to(torch.uint8)
    return x


def _params(case):
    p = {"raw_capacity": case.get("raw_capacity", 1 << 22)}
    if case.get("baseline") == "mean":
        p["baseline_mode"] = 1
    if case.get("rfi"):
        p["rfi"] = 1
    variant = case.get("variant", "plain")
    if variant == "subband":
        p["subband_chans"] = min(64, case["nchans"])
        p["subband_group"] = 8
    elif variant == "width_sigma":
        p["width_sigma"] = 1
    elif variant == "decimate":
        p["decimate"] = 16
    return p


def _out(capacity=CAND_CAPACITY):
    data, count = hp.new_cand_buf(capacity)
    data.zero_()
    return data, count


def _series(case, seed):
    """Dedispersed series as the pipeline meets them: int32 sums of 4096 channels,
    white noise, a slow drift, pulses of several widths."""
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 29)
    rng = np.random.RandomState(seed % (1 << 31))
    ndm, nout = case["ndm"], case["nsamps"]
    pitch = (nout + 3) // 4 * 4
    out = torch.zeros((ndm, pitch), dtype=torch.int32, device=dev)
    mean, sigma = 128.0 * 4096, 12.0 * 64.0
    t = torch.arange(nout, device=dev, dtype=torch.float32)
    drift = 0.5 * sigma * torch.sin(t * (2.0 * math.pi / 80000.0))
    pulses = [(rng.randint(0, ndm), rng.uniform(0.02, 0.98) * nout,
               math.exp(rng.uniform(0.0, math.log(400.0))), rng.uniform(9.0, 30.0))
              for _ in range(case["npulses"])]
    for d0 in range(0, ndm, 64):
        d1 = min(ndm, d0 + 64)
        v = torch.randn((d1 - d0, nout), device=dev, generator=gen) * sigma + mean + drift
        for d, c, w, snr in pulses:
            # strongest at its own trial, weaker and broader in the neighbouring ones
            for k in range(max(d0, d - 3), min(d1, d + 4)):
                ww = w * (1 + abs(k - d))
                v[k - d0] += snr * sigma / math.sqrt(ww) / (1 + abs(k - d)) * torch.exp(-((t - c) / ww) ** 2)
        out[d0:d1, :nout] = v.round_().to(torch.int32)
    return out


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.RandomState((seed * 31 + 7) % (1 << 31))
    if kind == "detect":
        # one channel: only the trial count and the widths of the plan are used
        plan = hp.Plan(1, 1500.0, -0.1, 49.152e-6, np.arange(case["ndm"], dtype=np.float32),
                       synth.widths_pow2(case["wmax"]), 6.0, **_params(case))
        return {"kind": kind, "plan": plan, "series": _series(case, seed),
                "nout": case["nsamps"], "out": _out()}
    if kind == "batch":
        files = workloads.batch(nfiles=case["nfiles"], seed0=case["seed0"], len_lo=case["len_lo"],
                                len_hi=case["len_hi"], dm_hi=case["dm_hi"], wmax=case["wmax"])
        plans, fbs, outs = [], [], []
        for i, w in enumerate(files):
            o = w.obs
            plan = hp.Plan(o.nchans, o.f_top, o.chan_bw, o.tsamp, w.dm_list, w.widths, w.threshold,
                           raw_capacity=1 << 20)
            plan.bind_workspace(o.nsamps)
            plans.append(plan)
            t_hi = plan.nout(o.nsamps) * o.tsamp
            fbs.append(_filterbank(o, seed * 64 + i,
                                   _pulses(o, rng, rng.randint(0, 11), case["dm_hi"], t_hi)))
            outs.append(_out(1 << 14))
        return {"kind": kind, "batch": hp.Batch(plans), "fbs": fbs, "outs": outs}
    obs = _obs(case)
    dms = _dm_list(case, obs)
    widths = synth.widths_pow2(case["wmax"])
    if kind == "stream":
        G, nb, ng = case["gulp"], case["nbeams"], case["ngulps"]
        plan = hp.Plan(obs.nchans, obs.f_top, obs.chan_bw, obs.tsamp, dms, widths, 6.0)
        gulps = []
        for b in range(nb):
            o = synth.Observation(nchans=obs.nchans, f_top=obs.f_top, chan_bw=obs.chan_bw,
                                  tsamp=obs.tsamp, nsamps=G * ng, mean=obs.mean, sigma=obs.sigma)
            x = _filterbank(o, seed * 64 + b, _pulses(o, rng, 2, case["dm_hi"], 0.6 * G * ng * o.tsamp))
            host = torch.empty(x.shape, dtype=torch.uint8, pin_memory=True)
            host.copy_(x)
            gulps.append([host[g * G:(g + 1) * G] for g in range(ng)])
        stream = hp.Stream(plan, nbeams=nb, gulp=G, cand_capacity=GULP_CANDS)
        state = {"kind": kind, "plan": plan, "stream": stream, "gulps": gulps, "G": G, "pushed": 0}
        for _ in range(2):      # the beams have been running: their tails are full
            _run_stream(state)
        return state
    plan = hp.Plan(obs.nchans, obs.f_top, obs.chan_bw, obs.tsamp, dms, widths, 6.0, **_params(case))
    plan.bind_workspace(obs.nsamps)
    t_hi = plan.nout(obs.nsamps) * obs.tsamp
    fb = _filterbank(obs, seed, _pulses(obs, rng, case["npulses"], case["dm_hi"], t_hi), case["stress"])
    state = {"kind": kind, "plan": plan, "fb": fb}
    if kind == "dedisperse":
        nout = plan.nout(obs.nsamps)
        state["out"] = torch.zeros((plan.ndm, (nout + 3) // 4 * 4), dtype=torch.int32, device=fb.device)
    else:
        state["out"] = _out(1 << 18 if case["stress"] else CAND_CAPACITY)
    return state


# ------------------------------------------------------------------ one pass
def _run_stream(state):
    """Push every beam's next gulps, poll every result; candidate times relative to
    the first sample of the pass, so that every pass returns the same table."""
    st, gulps, G = state["stream"], state["gulps"], state["G"]
    nb, ng = len(gulps), len(gulps[0])
    g0 = state["pushed"]
    for g in range(ng):
        for b in range(nb):
            st.push(b, gulps[b][g])
    state["pushed"] = g0 + ng
    got = {}
    while len(got) < nb * ng:
        info, cands = st.poll(-1)
        if info["status"] != 0:
            raise RuntimeError("gulp status %d" % info["status"])
        got[(info["beam"], info["gulp_index"] - g0)] = (info, cands)
    keys = sorted(got)
    base = g0 * G
    table = np.zeros((len(keys), GULP_CANDS), dtype=hp.CAND_DTYPE)
    for i, k in enumerate(keys):
        c = got[k][1]
        table[i, : c.size] = c
        for name in ("sample", "t_lo", "t_hi"):
            table[name][i, : c.size] -= base
    info = np.array([(k[0], k[1], got[k][0]["ncand"], got[k][0]["window_start"] - base,
                      got[k][0]["window_len"]) for k in keys], dtype=np.int64)
    return {"cands": table.view(np.uint8), "gulps": info}


def run(state):
    kind = state["kind"]
    if kind == "search":
        data, count = hp.hp_search(state["plan"], state["fb"], out=state["out"])
        return {"cands": data, "count": count}
    if kind == "dedisperse":
        return {"series": hp.hp_dedisperse(state["plan"], state["fb"], out=state["out"])}
    if kind == "detect":
        raw, nraw, sigma, mad = hp.hp_detect(state["plan"], state["series"], state["nout"],
                                             capacity=1 << 18)
        data, count = hp.hp_merge(state["plan"], raw, nraw, sigma, out=state["out"])
        return {"cands": data, "count": count, "nraw": nraw, "sigma": sigma, "mad": mad}
    if kind == "batch":
        outs = state["batch"].search_async(state["fbs"], outs=state["outs"])
        return {"cands": [d for d, _ in outs], "count": [c for _, c in outs]}
    return _run_stream(state)


# ------------------------------------------------------------------ the floor
def work(case):
    """Input bytes read once, results written once; the direct sums' additions, and
    per (trial, sample) one threshold test per width plus the prefix addition."""
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for w in workloads.batch(nfiles=case["nfiles"], seed0=case["seed0"], len_lo=case["len_lo"],
                                 len_hi=case["len_hi"], dm_hi=case["dm_hi"], wmax=case["wmax"]):
            o = w.obs
            nout = o.nsamps - _max_delay(o.nchans, 500.0, o.tsamp * 1e6, case["dm_hi"])
            b += o.nsamps * o.nchans
            f += w.ndm * nout * (o.nchans + w.nw + 1)
        return {"bytes": b, "flops": f}
    nw = int(math.log2(case["wmax"])) + 1
    if kind == "detect":
        return {"bytes": 4 * case["ndm"] * case["nsamps"],
                "flops": case["ndm"] * case["nsamps"] * (nw + 1)}
    if kind == "stream":
        n = case["nbeams"] * case["ngulps"] * case["gulp"]
        return {"bytes": n * case["nchans"], "flops": case["ndm"] * n * (case["nchans"] + nw + 1)}
    nout = case["nsamps"] - _max_delay(case["nchans"], case["band"], case["tsamp_us"], case["dm_hi"])
    nbytes = case["nsamps"] * case["nchans"]
    if kind == "dedisperse":
        return {"bytes": nbytes + 4 * case["ndm"] * nout, "flops": case["ndm"] * nout * case["nchans"]}
    per = case["nchans"]
    if case["variant"] == "subband":     # partial sums of groups of 8 trials, then 64 per trial
        per = case["nchans"] / 8 + math.ceil(case["nchans"] / 64)
    return {"bytes": nbytes, "flops": case["ndm"] * nout * (per + nw + 1)}


# ------------------------------------------------------------------ 64 bits
def exact(case, seed):
    """The dedispersed sums and the per-trial statistics, from their definitions."""
    if case["kind"] == "dedisperse":
        return _exact_dedisperse(case, seed)
    if case["kind"] == "detect":
        return _exact_detect(case, seed)
    return None     # candidate lists: whole numbers and one rounded S/N each


def _exact_dedisperse(case, seed):
    if case["ndm"] * case["nsamps"] * case["nchans"] > 1 << 38:
        return None
    state = prepare(case, seed)
    fb, dms = state["fb"], state["plan"].dm_list.astype(np.float64)
    obs = _obs(case)
    f = obs.f_top + np.arange(obs.nchans, dtype=np.float64) * obs.chan_bw
    delay = np.rint(K_DM * dms[:, None] * (1.0 / (f * f) - 1.0 / (obs.f_top * obs.f_top))[None, :]
                    / obs.tsamp).astype(np.int64)
    nout = obs.nsamps - int(delay.max())
    total = torch.zeros((len(dms), nout), dtype=torch.int64, device=fb.device)
    dev = torch.from_numpy(delay).to(fb.device)
    t = torch.arange(nout, device=fb.device)
    for c in range(obs.nchans):
        total += fb[:, c].contiguous().to(torch.int64)[dev[:, c, None] + t[None, :]]
    out = torch.zeros((len(dms), (nout + 3) // 4 * 4), dtype=torch.int64, device=fb.device)
    out[:, :nout] = total
    return {"series": out}


def _lower_median5(x):
    """Medians of five along the last axis, a trailing group's lower median."""
    n = x.shape[-1]
    full = x[..., : n // 5 * 5].reshape(*x.shape[:-1], n // 5, 5).sort(-1).values[..., 2]
    if n % 5 == 0:
        return full
    rest = x[..., n // 5 * 5:].sort(-1).values[..., (n % 5 - 1) // 2]
    return torch.cat([full, rest[..., None]], -1)


def _exact_detect(case, seed):
    series = _series(case, seed)
    n = case["nsamps"]
    win = int(math.floor(2.0 / 49.152e-6 + 0.5))
    sigma, mad = [], []
    t = torch.arange(n, device=series.device)
    for d0 in range(0, case["ndm"], 32):
        D = series[d0:d0 + 32, :n].to(torch.int64)
        if case["baseline"] == "mean":
            H = win // 2
            P = torch.nn.functional.pad(D.cumsum(-1), (1, 0))
            lo, hi = (t - H).clamp(min=0), (t + H + 1).clamp(max=n)
            b = torch.div(P[:, hi] - P[:, lo], (hi - lo)[None, :], rounding_mode="floor")
        else:
            m, q = D, 1
            while q * 5 <= win:
                m, q = _lower_median5(m), q * 5
            u = t - (q - 1) // 2
            j = torch.div(u, q, rounding_mode="floor").clamp(0, m.shape[-1] - 1)
            k = (j + 1).clamp(max=m.shape[-1] - 1)
            frac = torch.where((u < 0) | (j == k), torch.zeros_like(u), u - j * q)
            b = m[:, j] + torch.div((m[:, k] - m[:, j]) * frac[None, :], q, rounding_mode="floor")
        y = (D - b).abs().sort(-1).values[:, (n - 1) // 2]
        mad.append(y)
        sigma.append(1.482602218505602 * y.to(torch.float64))
    return {"cands": None, "count": None, "nraw": None, "sigma": torch.cat(sigma), "mad": torch.cat(mad)}

"""The work a user of this library has it do, as timed cases.

``listed`` holds the cases, ``draw`` gives further ones of the same ranges,
``prepare`` makes what a user's program has in hand (inputs on the device, the
plan, output and workspace buffers), ``run`` is one pass through the public
entry points, ``work`` the bytes and operations the path cannot do without and
``exact`` the same outputs from plain torch in 64 bits.

A case is one plan shape (channels, samples, DM trials, widths, mode, smoothing,
zapping) and the call made on it:

  search      Plan.search: the whole path on device buffers
  host        sps_search_host: the same from pinned host memory and back
  batch       Batch.launch: several beams in one graph launch
  noalloc     sps_dedisperse_noalloc (single-channel kernel, no workspace)
  snr         sps_snr on de-dispersed rows already on the device
  steps       sps_subband_step1, then sps_subband_step2 (Y returned as well)

Ranges: 37..1536 channels over 1250-1550 MHz at 81.92 us, 1000..12500 output
samples (rows of 57000..70000 in the long-row S/N case), 16..4096 DM trials in
steps of 0.1..2, one to seven boxcar widths, 8..48 subbands of 12..96 channels.
"""
import numpy as np
import torch

import paper_1811_04165_gb300 as sps

F_LO, F_HI, T_SAMP = 1250.0, 1550.0, 81.92e-6
K_DM = 4.148808e3
POW2 = "1,2,4,8,16,32,64"


def _case(kind, channels, n_t, n_dms, step, widths=POW2, subbands=0, coarse=0, decimate=False, zap=0, beams=1):
    return {"kind": kind, "channels": channels, "n_t": n_t, "n_dms": n_dms, "step": step, "widths": widths,
            "subbands": subbands, "coarse": coarse, "decimate": decimate, "zap": zap, "beams": beams}


def listed():
    return [
        # the smallest search: 64 channels, 32 trials, as a quick look or a check of the chain does; launches count
        {"name": "tiny_search", **_case("search", 64, 4096, 32, 2.0, "1,2,4,8")},
        # odd sizes everywhere and widths that are no powers of two (another instrument's settings)
        {"name": "ragged_search", **_case("search", 389, 7013, 517, 0.31, "1,3,5,11,23,47")},
        # one beam of the coarser channelisation of the batched and served mix
        {"name": "beam384_search", **_case("search", 384, 12500, 1024, 0.3)},
        # one Apertif-shaped beam, 1.024 s of data: the library's ordinary work
        {"name": "beam_search", **_case("search", 1536, 12500, 2048, 0.2)},
        # the most trials a served beam has
        {"name": "beam4096_search", **_case("search", 1536, 12500, 4096, 0.1)},
        # the ordinary beam by the two-step path
        {"name": "beam_subband", **_case("search", 1536, 12500, 2048, 0.2, subbands=32, coarse=64)},
        # the two steps called one by one, on a smaller beam with other subbands
        {"name": "steps384", **_case("steps", 384, 12500, 768, 0.4, subbands=16, coarse=24)},
        # decimating downsampling (AMBER's factors) with 5 % of the channels zapped for interference
        {"name": "decimate_zap", **_case("search", 1536, 12500, 512, 0.4, "10,20,40,80,160,320,640,1280,2560",
                                         decimate=True, zap=5)},
        # the ordinary beam from pinned host memory, results back on the host
        {"name": "beam_host", **_case("host", 1536, 12500, 2048, 0.2)},
        # beams of both channelisations with uneven trial counts, steps and widths in one graph launch
        {"name": "batch8", **_case("batch", 1536, 12500, 1024, 0.3, beams=8)},
        # de-dispersion for a caller that cannot allocate: the single-channel kernel
        {"name": "noalloc_dedisperse", **_case("noalloc", 1536, 12500, 768, 0.2)},
        # S/N of rows longer than a block's shared memory (5.7 s of data)
        {"name": "snr_long_rows", **_case("snr", 384, 70000, 384, 0.2)},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["subband"] * 3 + ["decimate"] * 2 + ["host", "batch", "noalloc", "snr", "steps"])
    widths = rng.choice([POW2, "1,2,4,8", "1,2,4,8,16,32", "1", "1,3,5,11,23,47", "1,2,3,6,12,25,50"])
    step = round(rng.uniform(0.1, 0.5), 2)
    n_t = rng.choice([12500, _log_int(rng, 1000, 12500), _log_int(rng, 1000, 12500)])
    channels = rng.choice([384, 1536, _log_int(rng, 37, 1536)])
    n_dms = max(16, min(_log_int(rng, 16, 4096), int(820 / step)))
    if kind == "snr":
        return _case("snr", 384, rng.choice([4 * _log_int(rng, 14250, 17500), n_t]),
                     _log_int(rng, 32, 512), step, rng.choice([POW2, "1,2,4,8,16"]))
    if kind in ("subband", "steps"):
        subbands = rng.choice([8, 16, 32, 48])
        per = _log_int(rng, 12, 96 if subbands < 32 else 1536 // subbands)
        coarse = _log_int(rng, 2, 64)
        fine = rng.choice([8, 16, 24, 32])
        return _case("steps" if kind == "steps" else "search", subbands * per, n_t, coarse * fine, step,
                     "1" if kind == "steps" else widths, subbands=subbands, coarse=coarse)
    if kind == "decimate":
        return _case("search", channels, n_t, n_dms, step, rng.choice(["10,20,40,80,160,320", "1,5,25,125", "10,100,1000"]),
                     decimate=True, zap=rng.choice([0, 5, 10]))
    if kind == "noalloc":
        n_dms = min(n_dms, int(409.6 / step))
    if kind == "batch":
        return _case("batch", 1536, n_t, _log_int(rng, 64, 1024), step, beams=rng.choice([2, 4, 8]))
    return _case(kind, channels, n_t, n_dms, step, widths, zap=rng.choice([0, 0, 0, 5]) if kind == "search" else 0)


def _beams(case):
    """The plan shapes of a case: itself, or a batch's beams (alternately the full and a quarter of the channels,
    trials, steps and width counts uneven)."""
    if case["kind"] != "batch":
        return [case]
    out = []
    for b in range(case["beams"]):
        n_dms = max(16, case["n_dms"] * (2 + (3 * b) % 5) // 4 // 16 * 16)
        k = 1 + (5 * b + 3) % 7
        out.append(_case("search", case["channels"] // (1 + 3 * (b % 2)), case["n_t"], n_dms,
                         round(case["step"] * (0.5 + 0.25 * (b % 4)), 3), ",".join(POW2.split(",")[:k])))
    return out


def _dms(c):
    return c["step"] * np.arange(c["n_dms"], dtype=np.float64)


def _widths(c):
    return [int(w) for w in c["widths"].split(",")]


def _zap(c):
    if not c["zap"]:
        return None
    rng = np.random.Generator(np.random.PCG64(c["channels"]))
    return (rng.random(c["channels"]) < c["zap"] / 100.0).astype(np.uint8)


def _coarse_dms(c):
    return _dms(c)[::c["n_dms"] // c["coarse"]].copy()


def _plan(c):
    kw = dict(smoothing=sps.SMOOTH_DECIMATE if c["decimate"] else sps.SMOOTH_SLIDING, zap=_zap(c))
    if c["subbands"]:
        kw.update(mode=sps.MODE_SUBBAND, n_subbands=c["subbands"], coarse_dms=_coarse_dms(c))
    return sps.Plan(c["channels"], F_LO, F_HI, T_SAMP, c["n_t"], _dms(c), _widths(c), **kw)


def _freqs(channels):
    return F_LO + (np.arange(channels, dtype=np.float64) + 0.5) * ((F_HI - F_LO) / channels)


def _filterbank(c, n_in, pitch, seed):
    """Gaussian noise (mean 128, sd 16) with five dispersed pulses, rounded and clipped to bytes: the digitised sky
    a telescope delivers."""
    gen = torch.Generator(device="cuda").manual_seed(1 + 7919 * int(seed))
    rng = np.random.Generator(np.random.PCG64(17 + int(seed)))
    C = c["channels"]
    sky = torch.randn((C, n_in), generator=gen, device="cuda", dtype=torch.float32).mul_(16.0).add_(128.0)
    f = _freqs(C)
    sweep = K_DM * (f ** -2 - f[-1] ** -2) / T_SAMP
    rows = torch.arange(C, device="cuda")
    for _ in range(5):
        dm = rng.uniform(0.02, 0.98) * max(c["step"], _dms(c)[-1])
        width = 2 ** int(rng.integers(0, 6))
        amp = rng.uniform(6.0, 20.0) * 16.0 / np.sqrt(C * width)
        at = torch.from_numpy(np.floor(rng.uniform(0, max(1, c["n_t"] - 64)) + dm * sweep).astype(np.int64)).cuda()
        for k in range(width):
            sky[rows, torch.clamp(at + k, max=n_in - 1)] += amp
    x = torch.zeros((C, pitch), dtype=torch.uint8, device="cuda")
    x[:, :n_in] = sky.round_().clamp_(0, 255).to(torch.uint8)
    return x


def _rows(c, seed):
    """De-dispersed rows as the search leaves them: sums of `channels` noise bytes, a pulse in some rows."""
    gen = torch.Generator(device="cuda").manual_seed(3 + 7919 * int(seed))
    C = c["channels"]
    d = torch.randn((c["n_dms"], c["n_t"]), generator=gen, device="cuda", dtype=torch.float32)
    d.mul_(16.0 * C ** 0.5).add_(128.0 * C)
    rng = np.random.Generator(np.random.PCG64(29 + int(seed)))
    for i in range(0, c["n_dms"], 7):
        w, t = 2 ** int(rng.integers(0, 6)), int(rng.integers(0, max(1, c["n_t"] - 64)))
        d[i, t:t + w] += rng.uniform(6.0, 20.0) * 16.0 * (C / w) ** 0.5
    return d.round_().clamp_(0, 255 * C).to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        plans = [_plan(c) for c in _beams(case)]
        xs = [_filterbank(c, p.input_samples, p.pitch, seed + 101 * b) for b, (c, p) in enumerate(zip(_beams(case), plans))]
        return {"kind": kind, "batch": sps.Batch(plans, xs)}
    plan = _plan(case)
    s = {"kind": kind, "plan": plan}
    if kind == "snr":
        s["out"] = plan.alloc_outputs()
        s["out"]["D"].copy_(_rows(case, seed))
        return s
    s["x"] = _filterbank(case, plan.input_samples, plan.pitch, seed)
    if kind == "noalloc":
        cfg = plan.config
        cfg.brute = sps.DedispConfig(4, 16, 8, 1, 16, 0)
        plan.config = cfg
        s["D"] = torch.empty((plan.n_dms, plan.n_samples), dtype=torch.int32, device="cuda")
        return s
    s["ws"] = plan.workspace()
    if kind == "steps":
        s["Y"] = torch.zeros(plan.y_shape, dtype=torch.int16, device="cuda").view(torch.uint16)
        s["D"] = torch.empty((plan.n_dms, plan.n_samples), dtype=torch.int32, device="cuda")
        return s
    s["out"] = plan.alloc_outputs()
    if kind == "host":
        s["x_host"] = s["x"].cpu().pin_memory()
        shape = (plan.n_widths, plan.n_dms)
        s["snr"] = torch.empty(shape, dtype=torch.float64).pin_memory()
        s["peak_t"] = torch.empty(shape, dtype=torch.int32).pin_memory()
        s["peak_val"] = torch.empty(shape, dtype=torch.int32).pin_memory()
        s["best"] = torch.empty(4, dtype=torch.int32).pin_memory()
    return s


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].launch()
        return state["batch"].outs
    plan = state["plan"]
    if kind == "search":
        return plan.search(state["x"], out=state["out"], workspace=state["ws"])
    if kind == "host":
        o = state["out"]
        sps.sps_search_host(plan, state["x_host"], state["x"], o["D"], o["snr"], o["peak_t"], o["peak_val"], o["best"],
                            state["snr"], state["peak_t"], state["peak_val"], state["best"], workspace=state["ws"])
        return {"D": o["D"], "snr": state["snr"], "peak_t": state["peak_t"], "peak_val": state["peak_val"],
                "best": state["best"]}
    if kind == "snr":
        o = state["out"]
        sps.sps_snr(plan, o["D"], o["snr"], o["peak_t"], o["peak_val"], o["best"])
        return {k: o[k] for k in ("snr", "peak_t", "peak_val", "best")}
    if kind == "noalloc":
        sps.sps_dedisperse_noalloc(plan, state["x"], state["D"])
        return {"D": state["D"]}
    sps.sps_subband_step1(plan, state["x"], state["Y"], workspace=state["ws"])
    sps.sps_subband_step2(plan, state["Y"], state["D"])
    return {"Y": state["Y"].view(torch.int16)[:, :, :plan.step1_samples], "D": state["D"]}


def _round(v):
    return np.floor(v + 0.5).astype(np.int64)


def _tables(c):
    """Delay tables in samples: brute force [trials][channels], or step one [coarse][channels] and step two
    [trials][subbands]."""
    f = _freqs(c["channels"])
    if not c["subbands"]:
        return _round(_dms(c)[:, None] * (K_DM * (1.0 / (f * f) - 1.0 / (f[-1] * f[-1])) / T_SAMP)[None, :]), None
    per = c["channels"] // c["subbands"]
    top = np.repeat(f[per - 1::per], per)
    d1 = _round(_coarse_dms(c)[:, None] * (K_DM * (1.0 / (f * f) - 1.0 / (top * top)) / T_SAMP)[None, :])
    ft = f[per - 1::per]
    d2 = _round(_dms(c)[:, None] * (K_DM * (1.0 / (ft * ft) - 1.0 / (f[-1] * f[-1])) / T_SAMP)[None, :])
    return d1, d2


def work(case):
    bytes_, ops = 0, 0
    for c in _beams(case):
        cells = c["n_dms"] * c["n_t"]
        table = 16 * len(_widths(c)) * c["n_dms"]
        boxcars = 3 * cells * len(_widths(c)) if not c["decimate"] else cells
        if case["kind"] == "snr":
            bytes_ += 4 * cells + table
            ops += boxcars
            continue
        d1, d2 = _tables(c)
        n_in = c["n_t"] + int(d1.max()) + (int(d2.max()) if d2 is not None else 0)
        bytes_ += c["channels"] * n_in + 4 * cells
        if c["subbands"]:
            n_1 = c["n_t"] + int(d2.max())
            ops += c["coarse"] * n_1 * c["channels"] + cells * c["subbands"]
            if case["kind"] == "steps":
                bytes_ += 2 * c["coarse"] * c["subbands"] * n_1
        else:
            ops += cells * c["channels"]
        if case["kind"] not in ("noalloc", "steps"):
            bytes_ += table
            ops += boxcars
    return {"bytes": bytes_, "flops": ops}


def _shift_sum(rows, delays, n_out):
    """sum over channels c of rows[c][t + delays[i][c]] for t < n_out, in 64-bit integers."""
    out = torch.zeros((delays.shape[0], n_out), dtype=torch.int64, device=rows.device)
    d = torch.from_numpy(np.ascontiguousarray(delays.T)).to(rows.device)
    for c in range(rows.shape[0]):
        out += rows[c].unfold(0, n_out, 1)[d[c]].to(torch.int64)
    return out


def _table_exact(c, D):
    """S/N, first peak and peak value of every (width, trial), in 64 bits."""
    P = torch.zeros((D.shape[0], D.shape[1] + 1), dtype=torch.int64, device=D.device)
    torch.cumsum(D, 1, out=P[:, 1:])
    snr, pt, pv = [], [], []
    for w in _widths(c):
        if c["decimate"]:
            n = D.shape[1] // w
            B = P[:, w:n * w + 1:w] - P[:, 0:(n - 1) * w + 1:w]
        else:
            B = P[:, w:] - P[:, :-w]
        m = B.max(1, keepdim=True).values
        at = torch.arange(B.shape[1], device=D.device)[None, :]
        first = torch.where(B == m, at, B.shape[1]).min(1).values
        # moments about an integer near the mean keep the sums exact, or nearly so, in 64 bits
        n = B.shape[1]
        z = (B - B[:, :1]).double()
        mean = z.mean(1, keepdim=True)
        var = (z - mean).square().mean(1)
        top = (m - B[:, :1]).double()[:, 0] - mean[:, 0]
        snr.append(torch.where(var > 0, top / var.clamp(min=1e-300).sqrt(), torch.zeros_like(var)))
        pt.append(first * w if c["decimate"] else first)
        pv.append(m[:, 0])
    return torch.stack(snr), torch.stack(pt).to(torch.int32), torch.stack(pv).to(torch.int32)


def exact(case, seed):
    outs = []
    for b, c in enumerate(_beams(case)):
        Y = None
        if case["kind"] == "snr":
            D = _rows(c, seed).to(torch.int64)
        else:
            d1, d2 = _tables(c)
            n_1 = c["n_t"] + (int(d2.max()) if d2 is not None else 0)
            n_in = n_1 + int(d1.max())
            x = _filterbank(c, n_in, (n_in + 15) // 16 * 16, seed + 101 * b if case["kind"] == "batch" else seed)
            if c["zap"]:
                x[torch.from_numpy(_zap(c)).cuda() != 0] = 0
            if c["subbands"]:
                per, fine = c["channels"] // c["subbands"], c["n_dms"] // c["coarse"]
                Y = torch.stack([_shift_sum(x[s * per:(s + 1) * per], d1[:, s * per:(s + 1) * per], n_1)
                                 for s in range(c["subbands"])], 1).to(torch.int32)
                D = torch.cat([_shift_sum(Y[k], d2[k * fine:(k + 1) * fine], c["n_t"]) for k in range(c["coarse"])])
            else:
                D = _shift_sum(x, d1, c["n_t"])
        if case["kind"] == "noalloc":
            return {"D": D.to(torch.int32)}
        if case["kind"] == "steps":
            return {"Y": Y.to(torch.int16), "D": D.to(torch.int32)}
        snr, pt, pv = _table_exact(c, D)
        # the detection is an argmax over the table, with ties by index: no value of its own
        o = {"snr": snr, "peak_t": pt, "peak_val": pv, "best": None}
        if case["kind"] != "snr":
            o["D"] = D.to(torch.int32)
        outs.append(o)
    return outs if case["kind"] == "batch" else outs[0]

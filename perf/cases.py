"""Cases that the library's speed is measured on: the calls of a dedispersion pipeline.

A case is one call sequence of include/dd.h's path through the Python binding, on a block
of synthetic filterbank data:

  step     channel statistics, dedispersion and boxcar S/N of a uint8 block (unit weights,
           exact int32 sums), as a search runs it
  fused    channel statistics and the fused dedispersion + boxcar call
  series   dedispersion alone with per-channel weights (fp32 sums)
  detect   channel statistics and boxcar S/N of a dedispersed series that is in hand
  batch    one block of many beams (dedispersion, statistics, boxcar) through a Batch
  train    forward and backward of DDFunction with learnable per-tap weights

Bands are those of synth/filterbank.py and bench.py: plain (64 channels, 1 ms), craft
(336 x 1 MHz, 1 ms) and low (1024 channels, 700-1000 MHz, 64 us).  Times of maxima are
returned where the sums that decide them are exact (integers, or fp32 holding whole
counts) or the series is an input.
"""
import math

import numpy as np
import torch

import paper_1301_3968_gb300 as dd

KDM = 4.15
# nchan, lowest edge (MHz), channel width (MHz), sampling time (ms)
BANDS = {"plain": (64, 1200.0, 4.6875, 1.0), "craft": (336, 1130.0, 1.0, 1.0),
         "low": (1024, 700.0, 300.0 / 1024.0, 0.064)}


# ----------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest block a user runs: launches and latency (bench.py's plain block)
        dict(name="plain_step", kind="step", band="plain", nsamp=4096, offset=0, ndm=128, dm_max=500.0,
             list="linear", wlo=1, whi=16),
        # one telescope beam of 8-bit data, ragged length, the direct integer sums
        dict(name="beam_step", kind="step", band="craft", nsamp=24001, offset=0, ndm=1500, dm_max=2000.0,
             list="rule", wlo=1, whi=32),
        # one chunk of the low-band stream: a window of a longer buffer, long tap runs
        dict(name="lowband_chunk", kind="step", band="low", nsamp=134980 + 65536, offset=40001, ndm=8192,
             dm_max=2000.0, list="linear", wlo=1, whi=256),
        # low-band detections only, the series not stored
        dict(name="lowband_fused", kind="fused", band="low", in_type="u8", nsamp=60000, ndm=1500, dm_max=366.0,
             list="linear", wlo=1, whi=64),
        # an 8-bit recording kept as float32 counts, detections only
        dict(name="counts_fused", kind="fused", band="craft", in_type="f32", nsamp=20001, ndm=1024,
             dm_max=1500.0, list="rule", wlo=1, whi=32),
        # the headline block of bench.py: fp32 data, weights by spectral index
        dict(name="craft_series", kind="series", band="craft", in_type="f32", nsamp=65536, ndm=4096,
             dm_max=4000.0, list="rule"),
        # 8-bit data with the same weights, a shorter and ragged block
        dict(name="weighted_u8", kind="series", band="craft", in_type="u8", nsamp=30011, ndm=700,
             dm_max=3000.0, list="rule"),
        # the detection stage of the headline block
        dict(name="craft_detect", kind="detect", band="craft", in_type="f32", nsamp=65536, ndm=4096,
             dm_max=4000.0, list="rule", widths="run", whi=32),
        # octave widths on integer sums, as a coarse search uses them
        dict(name="octave_detect", kind="detect", band="craft", in_type="u8", nsamp=24001, ndm=1500,
             dm_max=2000.0, list="rule", widths="octave", whi=512),
        # a block of unevenly sized beams in one launch (lower end of bench.py's batch)
        dict(name="beams_block", kind="batch", band="craft", nbeams=12, nsamp=16384, ndm=512, dm_max=1000.0,
             grow=1.06, whi=32),
        # a training step on bench.py's differentiable block: 32 learnable taps
        dict(name="train_block", kind="train", band="craft", nsamp=16384, ndm=1024, dm_max=2000.0, taps=32),
        # the weight-learning loop of one trial
        dict(name="train_trial", kind="train", band="plain", nsamp=1024, ndm=1, dm_max=150.0, taps=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "fused", "series", "detect", "batch", "train"])
    if kind == "batch":
        nsamp = _log(rng, 8192, 30000)
        return dict(kind=kind, band="craft", nbeams=rng.randint(2, 16), nsamp=nsamp, ndm=_log(rng, 64, 900),
                    dm_max=min(rng.uniform(300.0, 3000.0), _dm_for("craft", nsamp // 2)),
                    grow=rng.uniform(1.0, 1.08), whi=rng.randint(8, 40))
    if kind == "train":
        band = rng.choice(["plain", "craft"])
        nsamp, ndm = _log(rng, 1024, 14000), _log(rng, 1, 900)
        dm = 0.0 if ndm == 1 else min(rng.uniform(100.0, 2000.0), _dm_for(band, nsamp // 2))
        return dict(kind=kind, band=band, nsamp=nsamp, ndm=ndm, dm_max=max(dm, 50.0), taps=rng.randint(4, 48))
    band = rng.choice(["plain", "craft", "craft", "low"])
    if band == "low":
        # the low-band lists keep about the bench's DM spacing (0.24)
        nsamp, ndm = _log(rng, 20000, 150000), _log(rng, 100, 2500)
        dm = min(ndm * rng.uniform(0.15, 0.3), _dm_for(band, int(0.7 * nsamp)))
        c = dict(kind=kind, band=band, nsamp=nsamp, ndm=ndm, dm_max=dm, list="linear")
        wmax = 256
    else:
        nsamp, ndm = _log(rng, 3000, 60000), _log(rng, 40, 3000)
        dm = min(rng.uniform(300.0, 4000.0), _dm_for(band, int(0.7 * nsamp)))
        c = dict(kind=kind, band=band, nsamp=nsamp, ndm=ndm, dm_max=dm, list=rng.choice(["rule", "linear"]))
        wmax = 64
    if kind == "step":
        c.update(offset=rng.choice([0, rng.randint(1, 5000)]), wlo=1, whi=rng.randint(4, wmax))
    elif kind == "fused":
        c.update(in_type="u8" if band == "low" else rng.choice(["u8", "f32"]), wlo=1, whi=rng.randint(4, wmax))
    elif kind == "series":
        c.update(in_type=rng.choice(["u8", "f32"]))
        if band == "low":  # weights on short tap runs: the low end of the DM range
            c.update(ndm=min(ndm, 400), dm_max=min(dm, 60.0))
    else:
        c.update(in_type="u8" if band == "low" else rng.choice(["u8", "f32"]),
                 widths=rng.choice(["run", "run", "octave"]),
                 whi=rng.randint(8, wmax))
    return c


def _dm_for(band, dmax):
    """The DM whose sweep across the band is dmax samples."""
    C, lo, df, dt = BANDS[band]
    a, b = lo / 1000.0, (lo + C * df) / 1000.0
    return dmax * dt / (KDM * (a ** -2 - b ** -2))


# ----------------------------------------------------------------------------- tables

def _trials(band, ndm, dm_max, how):
    """Trial DMs from 0: evenly spaced, or growing as the trial rule's continuous form
    dDM/dn ~ sqrt(DM^2 + b^2) does, DM = b sinh(a n), b the DM whose smear is one sample."""
    if ndm == 1:
        return np.array([float(dm_max)])
    if how == "linear":
        return np.linspace(0.0, dm_max, ndm)
    C, lo, df, dt = BANDS[band]
    nu = (lo + (np.arange(C) + 1) * df) / 1000.0
    b = math.sqrt(2.0) * dt / (2.0 * KDM * df / 1000.0) / float(np.mean(nu ** -3))
    return b * np.sinh(np.linspace(0.0, math.asinh(dm_max / b), ndm))


def _tables(band, dms):
    """Start delays and tap counts of the band's channels (FP64, as include/dd.h states)."""
    C, lo, df, dt = BANDS[band]
    nu = (lo + (np.arange(C) + 1) * df) / 1000.0
    top = (lo + C * df) / 1000.0
    low = nu - df / 1000.0
    kd = KDM * np.asarray(dms)[:, None]
    delay = np.floor(kd * (1.0 / (nu * nu) - 1.0 / (top * top))[None, :] / dt).astype(np.int64)
    taps = np.maximum(1, np.ceil(kd * (1.0 / (low * low) - 1.0 / (nu * nu))[None, :] / dt)).astype(np.int64)
    return delay, taps


def _spectral(band):
    """Per-channel weights (nu / 1.298 GHz)^-1.4."""
    C, lo, df, _ = BANDS[band]
    return (((lo + (np.arange(C) + 0.5) * df) / 1000.0 / 1.298) ** -1.4).astype(np.float32)


def _widths(c):
    if c.get("widths") == "octave":
        return np.array([1 << i for i in range(int(math.log2(c["whi"])) + 1)], np.int32)
    return np.arange(c.get("wlo", 1), c["whi"] + 1, dtype=np.int32)


def _band(c, nsamp, in_type):
    C, lo, df, dt = BANDS[c["band"]]
    return dd.Band(C, lo, df, dt, nsamp, in_type)


def _t_out(c):
    d, n = _tables(c["band"], _trials(c["band"], c["ndm"], c["dm_max"], c.get("list", "rule")))
    return c["nsamp"] - int((d + (c["taps"] if c["kind"] == "train" else n)).max()) + 1


def _beams(c):
    """The beams of a batch: each `grow` times longer, with `grow` times the trials."""
    for i in range(c["nbeams"]):
        f = c["grow"] ** i
        yield dict(band=c["band"], kind="step", nsamp=int(c["nsamp"] * f), ndm=int(c["ndm"] * f),
                   dm_max=c["dm_max"], list="rule")


# ----------------------------------------------------------------------------- inputs

def _data(c, n, in_type, gen, counts=False):
    """Noise with three dispersed pulses, [nchan][n padded to 16 bytes]: uint8 N(128, 16^2),
    or fp32 N(0, 1), or fp32 whole counts N(0, 16^2)."""
    C, lo, df, dt = BANDS[c["band"]]
    q = 16 if in_type == "u8" else 4
    ld = (n + q - 1) // q * q
    sigma = 1.0 if in_type == "f32" and not counts else 16.0
    x = torch.randn((C, ld), generator=gen, device="cuda", dtype=torch.float32)
    u = torch.rand((3, 2), generator=gen, device="cuda").cpu().numpy()
    rows = torch.arange(C, device="cuda")[:, None]
    for k in range(3):
        d, t = _tables(c["band"], [c["dm_max"] * (0.2 + 0.7 * float(u[k, 0]))])
        t0 = int(0.2 * n * float(u[k, 1]))
        m = int(t.max()) + 1
        at = torch.from_numpy(d[0] + t0).cuda()[:, None] + torch.arange(m, device="cuda")[None, :]
        on = torch.arange(m, device="cuda")[None, :] <= torch.from_numpy(t[0]).cuda()[:, None]
        x[rows, at.clamp(max=ld - 1)] += 1.0 * on
    if in_type == "u8":
        return (x * sigma + 128.0).round().clamp(0, 255).to(torch.uint8)
    return (x * sigma).round() if counts else x


def _series(c, gen, t_out, int_off):
    """A dedispersed series' like: correlated noise of the trials' own scale, a few peaks."""
    d, n = _tables(c["band"], _trials(c["band"], c["ndm"], c["dm_max"], c["list"]))
    s = torch.from_numpy(n.sum(1).astype(np.float32)).cuda()[:, None]
    y = torch.randn((c["ndm"], t_out + 2), generator=gen, device="cuda", dtype=torch.float32)
    y = (y[:, 2:] + 0.5 * y[:, 1:-1] + 0.25 * y[:, :-2]) * s.sqrt()
    at = torch.randint(0, t_out, (c["ndm"], 4), generator=gen, device="cuda")
    y.scatter_add_(1, at, (5.0 * s.sqrt()).expand(-1, 4).contiguous())
    return (16.0 * y + 128.0 * s).round().clamp(min=0).minimum(255.0 * s).to(torch.int32) if int_off else y


def _weighted(plan, band):
    """Sets a weight per channel on every tap of the plan's default runs."""
    _, taps = plan.tables()
    k = np.arange(int(taps.max()))
    w = np.where(k[None, None, :] < taps[:, :, None], _spectral(band)[None, :, None], np.float32(0.0))
    plan.set_profiles(weights=w)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = dict(case=c)
    kind = c["kind"]
    if kind == "batch":
        plans, xs, outs, means, sds, peaks, args = [], [], [], [], [], [], []
        widths = _widths(c)
        for b in _beams(c):
            plans.append(dd.Plan(_band(b, b["nsamp"], "u8"), _trials(b["band"], b["ndm"], b["dm_max"], "rule")))
            xs.append(_data(b, b["nsamp"], "u8", gen))
            C, D = xs[-1].shape[0], b["ndm"]
            outs.append(torch.empty((D, b["nsamp"] - plans[-1].d_max), dtype=torch.int32, device="cuda"))
            means.append(torch.empty(C, dtype=torch.float64, device="cuda"))
            sds.append(torch.empty_like(means[-1]))
            peaks.append(torch.empty((D, len(widths)), dtype=torch.float32, device="cuda"))
            args.append(torch.empty((D, len(widths)), dtype=torch.int32, device="cuda"))
        batch = dd.Batch(plans)
        batch.bind(xs, outs)
        batch.bind_boxcar(widths, means, sds, peaks, args)
        s.update(batch=batch, plans=plans, outs=outs, peaks=peaks, args=args)
        return s
    n = c["nsamp"] + c.get("offset", 0)
    in_type = c.get("in_type", "u8" if kind == "step" else "f32")
    plan = dd.Plan(_band(c, c["nsamp"], in_type), _trials(c["band"], c["ndm"], c["dm_max"], c.get("list", "rule")))
    s.update(plan=plan)
    if kind == "train":
        K, (_, taps) = c["taps"], plan.tables()
        # learnable taps start as noise about one on each trial's own run
        w = torch.rand((c["ndm"], taps.shape[1], K), generator=gen, device="cuda") + 0.5
        on = torch.arange(K, device="cuda")[None, None, :] < torch.from_numpy(taps).cuda()[:, :, None]
        w = w * on
        plan.set_profiles(taps=np.full_like(taps, K), weights=np.ones(w.shape, np.float32))
        g = torch.randn((c["ndm"], c["nsamp"] - plan.d_max), generator=gen, device="cuda")
        x = _data(c, n, "f32", gen)
        s.update(x=x.requires_grad_(True), w=w.requires_grad_(True), g=g)
        return s
    if kind == "series" or (kind == "detect" and in_type == "f32"):
        _weighted(plan, c["band"])
    s.update(x=_data(c, n, in_type, gen, counts=kind == "fused"))
    if kind == "detect":
        s.update(series=_series(c, gen, c["nsamp"] - plan.d_max, in_type == "u8"))
    if kind != "series":
        s.update(widths=_widths(c))
    return s


# ----------------------------------------------------------------------------- the calls

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "batch":
        state["batch"].run()
        return state["outs"], state["peaks"], state["args"]
    plan, x, n = state["plan"], state["x"], c["nsamp"]
    if kind == "train":
        x.grad = state["w"].grad = None
        y = dd.DDFunction.apply(x, state["w"], plan, 0, n)
        y.backward(state["g"])
        return y.detach(), x.grad, state["w"].grad
    if kind == "series":
        return plan.dedisperse(x, nsamp=n)
    off = c.get("offset", 0)
    mean, sd = plan.channel_stats(x, t_offset=off, nsamp=n)
    if kind == "step":
        y = plan.dedisperse(x, t_offset=off, nsamp=n)
        peak, arg, _ = plan.boxcar_snr(y, state["widths"], mean, sd)
        return y, mean, sd, peak, arg
    if kind == "fused":
        peak, arg, _ = plan.dedisperse_boxcar(x, state["widths"], mean, sd, nsamp=n)
    else:
        peak, arg, _ = plan.boxcar_snr(state["series"], state["widths"], mean, sd)
    return mean, sd, peak, arg


# ----------------------------------------------------------------------------- work

def _work(c):
    C, kind = BANDS[c["band"]][0], c["kind"]
    T, D, n = _t_out(c), c["ndm"], c["nsamp"]
    esz = 1 if c.get("in_type", "u8" if kind == "step" else "f32") == "u8" else 4
    if kind == "train":
        K = c["taps"]
        # the input, the weights and the output's gradient in; the series and both gradients out
        return 4 * (2 * C * n + 2 * D * C * K + 2 * D * T), 6 * D * C * K * T
    nw = len(_widths(c)) if kind != "series" else 0
    # a trial needs at least one sum per channel and output (a weighted one a multiply too),
    # and a detection one difference and one comparison per width and output
    return (C * n * esz + (0 if kind == "fused" else 4 * D * T) + 8 * D * nw,
            (0 if kind == "detect" else (2 if kind == "series" else 1) * D * C * T) + 2 * D * nw * T)


def work(case):
    parts = [_work(dict(b, whi=case["whi"])) for b in _beams(case)] if case["kind"] == "batch" else [_work(case)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ----------------------------------------------------------------------------- 64 bits

def _windows(row, T):
    return row.as_strided((row.numel() - T + 1, T), (1, 1))


def _dedisperse64(x, delay, taps, w, T):
    """sum_c w_c sum_{k<n} x[c][t + delta + k] from 64-bit running sums."""
    D, C = delay.shape
    out = torch.zeros((D, T), dtype=torch.float64, device="cuda")
    a, b = torch.from_numpy(delay).cuda(), torch.from_numpy(delay + taps).cuda()
    step = max(1, (1 << 28) // T)
    for c in range(C):
        p = torch.zeros(x.shape[1] + 1, dtype=torch.float64, device="cuda")
        torch.cumsum(x[c].double(), 0, out=p[1:])
        v = _windows(p, T)
        for i in range(0, D, step):
            out[i:i + step].add_(v[b[i:i + step, c]] - v[a[i:i + step, c]], alpha=float(w[c]))
    return out


def _stats64(x):
    x = x.double()
    return x.mean(1), x.std(1, correction=0)


def _peaks64(y, widths, taps, w, mean, sd):
    """(largest boxcar sum - mean) / deviation per trial and width."""
    n = torch.from_numpy(taps).cuda().double()
    wc = torch.from_numpy(np.asarray(w, np.float64)).cuda()
    mu1 = (n * (wc * mean)[None, :]).sum(1)
    peaks = torch.empty((y.shape[0], len(widths)), dtype=torch.float64, device="cuda")
    for i in range(0, y.shape[0], 512):
        p = torch.zeros((min(512, y.shape[0] - i), y.shape[1] + 1), dtype=torch.float64, device="cuda")
        torch.cumsum(y[i:i + 512].double() - mu1[i:i + 512, None], 1, out=p[:, 1:])
        for j, wd in enumerate(widths):
            # |1_n * 1_w|^2: a trapezoid
            m = torch.minimum(n[i:i + 512], torch.full_like(n[i:i + 512], float(wd)))
            q = (m - 1) * m * (2 * m - 1) / 3 + m * m * ((n[i:i + 512] - float(wd)).abs() + 1)
            var = (q * ((wc * sd) ** 2)[None, :]).sum(1)
            peaks[i:i + 512, j] = (p[:, wd:] - p[:, :-wd]).amax(1) / var.sqrt()
    return peaks


def _train64(c, x, w, g):
    x, w, g = x.detach().double(), w.detach().double(), g.double()
    D, C, K = w.shape
    T = g.shape[1]
    delay, _ = _tables(c["band"], _trials(c["band"], D, c["dm_max"], "rule"))
    y = torch.empty((D, T), dtype=torch.float64, device="cuda")
    gw = torch.empty_like(w)
    gx = torch.zeros_like(x)
    at0 = torch.arange(C, device="cuda")[:, None] * x.shape[1] + torch.arange(T + K - 1, device="cuda")[None, :]
    gp = torch.zeros(T + 2 * (K - 1), dtype=torch.float64, device="cuda")
    for d in range(D):
        at = at0 + torch.from_numpy(delay[d]).cuda()[:, None]
        v = x.view(-1)[at].as_strided((C, K, T), (T + K - 1, 1, 1))
        y[d] = sum(w[d, :, k] @ v[:, k] for k in range(K))
        gw[d] = torch.stack([v[:, k] @ g[d] for k in range(K)], 1)
        gp[K - 1:K - 1 + T] = g[d]
        # gx[c][delta + m] += sum_k w[c][k] g[m - k]
        gx.view(-1).index_add_(0, at.view(-1), (w[d].flip(1) @ _windows(gp, T + K - 1)).view(-1))
    return y, gx, gw


def exact(case, seed):
    c, kind = case, case["kind"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if kind == "batch":
        peaks = []
        for b in _beams(c):
            x = _data(b, b["nsamp"], "u8", gen)[:, :b["nsamp"]]
            delay, taps = _tables(b["band"], _trials(b["band"], b["ndm"], b["dm_max"], "rule"))
            w = np.ones(delay.shape[1])
            y = _dedisperse64(x, delay, taps, w, _t_out(b))
            peaks.append(_peaks64(y, _widths(c), taps, w, *_stats64(x)))
        return [None] * c["nbeams"], peaks, [None] * c["nbeams"]
    dms = _trials(c["band"], c["ndm"], c["dm_max"], c.get("list", "rule"))
    delay, taps = _tables(c["band"], dms)
    n, off = c["nsamp"], c.get("offset", 0)
    in_type = c.get("in_type", "u8" if kind == "step" else "f32")
    if kind == "train":
        if 6.0 * c["ndm"] * taps.shape[1] * c["taps"] * c["nsamp"] > 2e12:
            return None
        K = c["taps"]
        w = torch.rand((c["ndm"], taps.shape[1], K), generator=gen, device="cuda") + 0.5
        w = w * (torch.arange(K, device="cuda")[None, None, :] < torch.from_numpy(taps).cuda()[:, :, None])
        g = torch.randn((c["ndm"], _t_out(c)), generator=gen, device="cuda")
        return _train64(c, _data(c, n, "f32", gen), w, g)
    weighted = kind == "series" or (kind == "detect" and in_type == "f32")
    w = _spectral(c["band"]) if weighted else np.ones(delay.shape[1])
    x = _data(c, n + off, in_type, gen, counts=kind == "fused")[:, off:off + n]
    T = _t_out(c)
    mean, sd = _stats64(x)
    # about 2e10 sums a second
    big = float(c["ndm"]) * delay.shape[1] * T > 1.5e11
    if kind == "detect":
        y = _series(c, gen, T, in_type == "u8")
    else:
        y = None if big else _dedisperse64(x, delay, taps, w, T)
    if kind == "series":
        return y
    peak = None if y is None else _peaks64(y, _widths(c), taps, w, mean, sd)
    if kind == "step":
        return None, mean, sd, peak, None
    return mean, sd, peak, None

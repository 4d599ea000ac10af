"""Row kernels (tap sums shared by the trials of a CTA): against the oracle at the edges of
tiles, trial blocks, shifts between trials and tap counts, and where a plan leaves them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dd():
    import torch
    from paper_1301_3968_gb300 import build
    build.build()
    import paper_1301_3968_gb300 as m
    torch.cuda.set_device(0)
    return m


def _tables(rng, D, C, steps, tap_sets, group):
    """Trials whose starts grow by a step of `steps` on each channel, and whose taps change
    every `group` trials."""
    delay = np.cumsum(rng.choice(steps, size=(D, C)), axis=0).astype(np.int32)
    delay -= delay.min(axis=0) - rng.integers(0, 9, size=C).astype(np.int32)
    taps = rng.choice(tap_sets, size=((D + group - 1) // group, C))
    return delay, np.repeat(taps, group, axis=0)[:D].astype(np.int32)


def _input(rng, kind, C, ld):
    if kind == "u8":
        return rng.integers(0, 256, size=(C, ld)).astype(np.uint8)
    return rng.standard_normal((C, ld)).astype(np.float32)


def _weights(rng, taps, group):
    """Per-tap weights that change with the taps."""
    w = rng.standard_normal(((taps.shape[0] + group - 1) // group, taps.shape[1], int(taps.max())))
    return np.repeat(w, group, axis=0)[:taps.shape[0]].astype(np.float32)


@pytest.mark.parametrize("kind", ["f32", "u8"])
@pytest.mark.parametrize("seed,C,D,t_out,t_off,steps,tap_sets,group,nch", [
    (1, 5, 48, 864, 0, [0, 1, 2], [1, 2, 3, 4], 48, 1),          # one full tile and block
    (2, 7, 49, 865, 3, [0, 1, 3], [4, 5, 6, 7], 24, 1),          # one past both
    (3, 3, 47, 863, 1, [0, 0, 5], [8, 9, 13], 47, 1),            # one short of both
    (4, 40, 100, 5000, 7, [0, 1, 2, 4], [1, 23, 27, 28], 16, 1),  # stages, shifts of every case
    (5, 33, 25, 2600, 2, [0, 30], [54, 61], 5, 1),               # far trials, long runs
    (6, 20, 31, 3600, 0, [0, 2], [3, 17], 8, 2),                 # two time chunks per CTA
    (7, 12, 2, 40, 5, [1], [31], 2, 1),                          # fewer trials than a warp sums
    (8, 6, 4000, 1800, 0, [0, 1], [2, 6], 400, 1),               # 16 warps per CTA
])
def test_weighted_rows_against_oracle(dd, kind, seed, C, D, t_out, t_off, steps, tap_sets, group, nch):
    import torch
    rng = np.random.default_rng(seed)
    delay, taps = _tables(rng, D, C, steps, tap_sets, group)
    T = t_out + int((delay + taps - 1).max())
    ld = (T + t_off + 15) // 16 * 16
    I = _input(rng, kind, C, ld)
    w = _weights(rng, taps, group)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, kind), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps, weights=w)
    if nch > 1:
        plan.set_schedule(nch, 2)
        assert plan.schedule()["nch"] == nch
    got = plan.dedisperse(torch.from_numpy(I).cuda(), t_offset=t_off, nsamp=T).cpu().numpy()
    assert plan.device_status() == 0
    assert got.shape == (D, t_out)
    rows = sorted(set(rng.integers(0, D, size=12).tolist() + [0, D - 1]))
    want = oracle.c_dedisperse(I, delay, taps, w=w, t_offset=t_off, nsamp=T, rows=rows)
    scale = oracle.c_abs_scale(I, delay, taps, w=w, t_offset=t_off, nsamp=T, rows=rows)
    assert (np.abs(got[rows] - want) <= 1e-5 * scale).all()


def test_rows_keep_nan_and_infinity_inside_runs(dd):
    """A NaN or infinite sample reaches exactly the outputs whose run holds it, as the sum
    over the run's own samples says."""
    import torch
    rng = np.random.default_rng(21)
    C, D, t_out = 9, 60, 1200
    delay, taps = _tables(rng, D, C, [0, 1, 2], [1, 2, 3, 5, 6, 7], 60)
    T = t_out + int((delay + taps - 1).max())
    I = _input(rng, "f32", C, (T + 3) // 4 * 4)
    bad = [(0, 100, np.nan), (3, 700, np.inf), (5, 901, -np.inf), (8, T - 1, np.nan)]
    for c, t, v in bad:
        I[c, t] = v
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "f32"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps)
    got = plan.dedisperse(torch.from_numpy(I).cuda(), nsamp=T).cpu().numpy()
    hit = np.zeros((D, t_out), bool)
    for c, t, _ in bad:
        for d in range(D):
            lo = t - delay[d, c] - taps[d, c] + 1
            hit[d, max(0, lo):max(0, t - delay[d, c] + 1)] = True
    np.testing.assert_array_equal(~np.isfinite(got), hit)


def test_device_weights_leave_the_rows(dd):
    """Weights from the device, which need not be shared, replace host weights that were; a
    batch bound before, and its graph, follow."""
    import torch
    rng = np.random.default_rng(31)
    C, T = 24, 3000
    plans, xs, outs, ws = [], [], [], []
    for D in (40, 33):
        delay, taps = _tables(rng, D, C, [0, 1], [3, 4], D)
        p = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "f32"), np.zeros(D))
        p.set_profiles(delay=delay, taps=taps, weights=np.full((D, C, 4), 0.5, np.float32))
        plans.append(p)
        xs.append(torch.from_numpy(_input(rng, "f32", C, T)).cuda())
        outs.append(torch.empty((D, T - p.d_max), device="cuda"))
        ws.append((delay, taps, rng.standard_normal((D, C, 4)).astype(np.float32)))
    batch = dd.Batch(plans)
    batch.bind(xs, outs)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    batch.capture(s)
    s.synchronize()
    first = [o.clone() for o in outs]
    for p, x, o in zip(plans, xs, first):
        assert torch.equal(p.dedisperse(x, nsamp=T), o)
    plans[0].set_weights(torch.from_numpy(ws[0][2]).cuda())
    torch.cuda.synchronize()
    for _ in range(2):  # the call that sees the new tables, and the graph made from them
        for o in outs:
            o.zero_()
        torch.cuda.synchronize()
        batch.replay(s)
        s.synchronize()
        assert torch.equal(outs[1], first[1])
        delay, taps, w = ws[0]
        I = xs[0].cpu().numpy()
        want = oracle.c_dedisperse(I, delay, taps, w=w, nsamp=T)
        scale = oracle.c_abs_scale(I, delay, taps, w=w, nsamp=T)
        assert (np.abs(outs[0].cpu().numpy() - want) <= 1e-5 * scale).all()


@pytest.mark.parametrize("seed,D,steps,w0,w1,parts", [
    (41, 100, [0, 1, 2], 1, 32, 0),
    (42, 49, [0, 1, 4], 5, 60, 7),
    (43, 1400, [0, 1], 1, 40, 0),      # 16 warps per CTA
    (44, 1400, [0, 1], 790, 835, 0),   # and a carry that leaves one row per warp
])
def test_fused_weighted_rows(dd, seed, D, steps, w0, w1, parts):
    """Fused = unfused, bit for bit."""
    import torch
    rng = np.random.default_rng(seed)
    C, t_out = 10, 5000
    delay, taps = _tables(rng, D, C, steps, [2, 3, 7], (D + 1) // 2)
    T = t_out + int((delay + taps - 1).max())
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "f32"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps, weights=_weights(rng, taps, (D + 1) // 2))
    x = torch.from_numpy(_input(rng, "f32", C, (T + 3) // 4 * 4)).cuda()
    mean, sd = plan.channel_stats(x, nsamp=T)
    widths = np.arange(w0, w1 + 1, dtype=np.int32)
    plan.test_set_fused_parts(parts)
    p0, a0, _ = plan.boxcar_snr(plan.dedisperse(x, nsamp=T), widths, mean, sd)
    p1, a1, _ = plan.dedisperse_boxcar(x, widths, mean, sd, nsamp=T)
    assert plan.device_status() == 0
    assert torch.equal(p0.view(torch.int32), p1.view(torch.int32)) and torch.equal(a0, a1)


@pytest.mark.parametrize("method", ["direct", "runlength"])
@pytest.mark.parametrize("seed,C,D,t_out,t_off,steps,tap_sets,group,nch", [
    (51, 8, 32, 1088, 0, [0, 1, 2], [1, 2, 3, 4], 32, 1),          # one full tile and block
    (52, 7, 33, 1089, 3, [0, 1, 9], [5, 6, 7, 8], 16, 1),          # one past both
    (53, 3, 31, 1087, 17, [0, 40], [64, 65], 31, 1),               # one short of both
    (54, 70, 100, 3000, 5, [0, 1, 2], [63, 64, 65, 66], 25, 1),    # four words' sums just fit, or two and two
    (55, 41, 40, 2500, 1, [0, 3], [128, 129], 20, 1),              # two and two, or none
    (56, 30, 37, 2200, 2, [0, 1], [254, 257], 37, 1),              # the longest runs
    (57, 9, 20, 600, 0, [0, 1], [258], 20, 1),                     # one past: the tap kernels
    (58, 21, 40, 4500, 0, [0, 2], [3, 200], 20, 2),                # two time chunks per CTA
    (59, 5, 1, 40, 9, [1], [2], 1, 1),                             # one trial: no sharing
    (60, 6, 6000, 1800, 0, [0, 1], [2, 6], 400, 1),                # 16 warps per CTA
])
@pytest.mark.parametrize("data", ["noise", "saturated"])
def test_packed_rows_bit_exact(dd, method, seed, C, D, t_out, t_off, steps, tap_sets, group, nch, data):
    """uint8 sums equal the oracle's, with every sample at 255 too (the largest half words)."""
    import torch
    rng = np.random.default_rng(seed)
    delay, taps = _tables(rng, D, C, steps, tap_sets, group)
    T = t_out + int((delay + taps - 1).max())
    ld = (T + t_off + 15) // 16 * 16
    I = _input(rng, "u8", C, ld) if data == "noise" else np.full((C, ld), 255, np.uint8)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "u8"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps)
    plan.set_method(method)
    if nch > 1:
        plan.set_schedule(nch, 3)
        assert plan.schedule()["nch"] == nch
    got = plan.dedisperse(torch.from_numpy(I).cuda(), t_offset=t_off, nsamp=T).cpu().numpy()
    assert plan.device_status() == 0
    rows = sorted(set(rng.integers(0, D, size=12).tolist() + [0, D - 1]))
    want = oracle.c_dedisperse(I, delay, taps, t_offset=t_off, nsamp=T, rows=rows)
    np.testing.assert_array_equal(got[rows].astype(np.int64), want)


@pytest.mark.parametrize("method", ["direct", "runlength"])
@pytest.mark.parametrize("seed,D,steps,w0,w1,parts,nch", [
    (71, 100, [0, 1, 2], 1, 32, 0, 1),
    (72, 49, [0, 1, 4], 5, 90, 7, 1),     # pruned width groups
    (73, 2400, [0, 1], 1, 256, 0, 1),     # 16 warps per CTA
    (74, 60, [0, 1], 960, 993, 5, 1),     # the longest carry a plan takes
    (75, 40, [0, 2], 1, 70, 4, 2),        # two time chunks per CTA
])
def test_fused_packed_rows(dd, method, seed, D, steps, w0, w1, parts, nch):
    """Fused = unfused, bit for bit, ties (constant channels) included."""
    import torch
    rng = np.random.default_rng(seed)
    C, t_out = 10, 6500
    delay, taps = _tables(rng, D, C, steps, [2, 3, 7], (D + 1) // 2)
    T = t_out + int((delay + taps - 1).max())
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "u8"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps)
    plan.set_method(method)
    if nch > 1:
        plan.set_schedule(nch, 4)
    I = np.clip(rng.normal(128, 3, size=(C, (T + 15) // 16 * 16)), 0, 255).astype(np.uint8)
    I[:, 2000:3500] = 128
    x = torch.from_numpy(I).cuda()
    mean, sd = plan.channel_stats(x, nsamp=T)
    widths = np.arange(w0, w1 + 1, dtype=np.int32)
    plan.test_set_fused_parts(parts)
    p0, a0, _ = plan.boxcar_snr(plan.dedisperse(x, nsamp=T), widths, mean, sd)
    p1, a1, _ = plan.dedisperse_boxcar(x, widths, mean, sd, nsamp=T)
    assert plan.device_status() == 0
    assert torch.equal(p0.view(torch.int32), p1.view(torch.int32)) and torch.equal(a0, a1)


@pytest.mark.parametrize("method", ["direct", "runlength"])
@pytest.mark.parametrize("seed,nch,w0,w1,parts", [
    (76, 1, 600, 634, 0),       # C = 633: a row per trial no longer leaves room for static variables
    (77, 1, 630, 635, 0),       # the first widths that take turns in one row per warp
    (78, 1, 660, 700, 6),
    (79, 1, 930, 993, 0),       # the longest carry
    (80, 2, 1240, 1260, 0),     # two time chunks, on either side of their line
    (81, 2, 1255, 1262, 7),
    (82, 2, 1970, 1985, 0),
])
def test_fused_packed_rows_of_wide_lists(dd, method, seed, nch, w0, w1, parts):
    """Sixteen warps per CTA and carries whose rows do not all fit its shared memory: fused =
    unfused, bit for bit."""
    import torch
    rng = np.random.default_rng(seed)
    C, t_out, D = 6, 6500, 2373
    delay, taps = _tables(rng, D, C, [0, 1], [2, 3, 7], 1184)
    T = t_out + int((delay + taps - 1).max())
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "u8"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps)
    plan.set_method(method)
    if nch > 1:
        plan.set_schedule(nch, 4)
    assert plan.schedule()["trials_per_cta"] == 32 // nch
    I = np.clip(rng.normal(128, 3, size=(C, (T + 15) // 16 * 16)), 0, 255).astype(np.uint8)
    I[:, 2000:3500] = 128
    x = torch.from_numpy(I).cuda()
    mean, sd = plan.channel_stats(x, nsamp=T)
    widths = np.arange(w0, w1 + 1, dtype=np.int32)
    plan.test_set_fused_parts(parts)
    p0, a0, _ = plan.boxcar_snr(plan.dedisperse(x, nsamp=T), widths, mean, sd)
    p1, a1, _ = plan.dedisperse_boxcar(x, widths, mean, sd, nsamp=T)
    assert plan.device_status() == 0
    assert torch.equal(p0.view(torch.int32), p1.view(torch.int32)) and torch.equal(a0, a1)


def test_batch_of_rows_and_taps(dd):
    """Beams of the row kernels (8 and 16 warps per CTA) and of the tap kernel in one batch, and
    the graph of it, equal the beams' own launches."""
    import torch
    rng = np.random.default_rng(81)
    C = 16
    plans, xs, outs = [], [], []
    for D, T, group in ((40, 2500, 40), (5000, 2600, 500), (30, 2300, 1)):
        delay, taps = _tables(rng, D, C, [0, 1], list(range(1, 20)), group)
        delay %= 60
        p = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "u8"), np.zeros(D))
        p.set_profiles(delay=delay, taps=taps)
        p.set_method("direct")
        plans.append(p)
        xs.append(torch.from_numpy(_input(rng, "u8", C, (T + 15) // 16 * 16)).cuda())
        outs.append(torch.zeros((D, T - p.d_max), dtype=torch.int32, device="cuda"))
    assert len({p.schedule()["trials_per_cta"] for p in plans}) == 3
    batch = dd.Batch(plans)
    batch.bind(xs, outs)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    batch.capture(s)
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    batch.replay(s)
    s.synchronize()
    for p, x, o in zip(plans, xs, outs):
        assert torch.equal(p.dedisperse(x, nsamp=p.band.nsamp), o)


def test_direct_calls_longer_than_the_band_go_in_pieces(dd):
    """A direct plan's prefix sums have room for its band's block; a longer call is summed in
    pieces, with the same results."""
    import torch
    rng = np.random.default_rng(91)
    C, D, T = 6, 40, 150000
    delay, taps = _tables(rng, D, C, [0, 1, 2], [2, 9], 20)
    I = _input(rng, "u8", C, T + 16)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, 3000, "u8"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps)
    plan.set_method("direct")
    got = plan.dedisperse(torch.from_numpy(I).cuda(), t_offset=5, nsamp=T).cpu().numpy()
    rows = [0, 17, D - 1]
    want = oracle.c_dedisperse(I, delay, taps, t_offset=5, nsamp=T, rows=rows)
    np.testing.assert_array_equal(got[rows].astype(np.int64), want)


@pytest.mark.parametrize("fused", [False, True])
def test_direct_plan_on_alternating_streams(dd, fused):
    """Two streams take one direct plan's calls in turn, with no synchronisation between them:
    each reads its own block's prefix sums."""
    import torch
    rng = np.random.default_rng(61)
    C, D, T = 64, 600, 40000
    delay, taps = _tables(rng, D, C, [0, 1], [2, 3], 48)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "u8"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps)
    assert plan.method == "direct"
    xs = [torch.from_numpy(_input(rng, "u8", C, T)).cuda() for _ in range(4)]
    m, sd = plan.channel_stats(xs[0])
    wl = np.arange(1, 9, dtype=np.int32)
    want = [plan.dedisperse(x) for x in xs]
    peak = plan.dedisperse_boxcar(xs[3], wl, m, sd)[0] if fused else None
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.default_stream(), torch.cuda.Stream()]
    for _ in range(3):
        got = []
        for x, s in zip(xs, streams):
            with torch.cuda.stream(s):
                if fused and s is streams[3]:
                    p = plan.dedisperse_boxcar(x, wl, m, sd)[0]
                else:
                    got.append(plan.dedisperse(x))
        torch.cuda.synchronize()
        for g, w in zip(got, want):
            assert torch.equal(g, w)
        if fused:
            assert torch.equal(p, peak)


@pytest.mark.parametrize("steps", [[0, 5, 9], [3, 9], [0, 1, 2, 9]])
@pytest.mark.parametrize("D", [2, 33])
def test_coarse_lists_against_oracle(dd, steps, D):
    """Lists whose neighbours share no, few or most windows, on either side of the rule for fp32
    rows; a list and its halves give the same bits where all are on one side."""
    import torch
    rng = np.random.default_rng(71)
    C, T = 12, 3000
    delay, taps = _tables(rng, D, C, steps, [2, 3, 7], 48)
    w = _weights(rng, taps, 48)
    I = _input(rng, "f32", C, T)
    x = torch.from_numpy(I).cuda()

    def run(sel):
        p = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "f32"), np.zeros(len(delay[sel])))
        p.set_profiles(delay=delay[sel], taps=taps[sel], weights=w[sel])
        return p.dedisperse(x, nsamp=T)

    got = run(slice(0, D))
    want = oracle.c_dedisperse(I, delay, taps, w=w, nsamp=T)
    scale = oracle.c_abs_scale(I, delay, taps, w=w, nsamp=T)
    assert (np.abs(got.cpu().numpy() - want) <= 1e-5 * scale).all()
    if steps == [3, 9]:  # no window is shared in any part
        n = got.shape[1]
        assert torch.equal(torch.cat([run(slice(0, D // 2))[:, :n], run(slice(D // 2, D))[:, :n]]), got)


def test_batch_of_one_wave_beams(dd):
    """Beams that alone leave SMs idle and together do not get smaller stages: the same sums, from
    the batch and from the plans afterwards."""
    import torch
    rng = np.random.default_rng(81)
    C, T, D = 40, 20000, 60
    plans, xs, outs, want = [], [], [], []
    for k in range(4):
        delay, taps = _tables(rng, D, C, [0, 1, 3], [1, 2, 5], 20)
        p = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "u8"), np.zeros(D))
        p.set_profiles(delay=delay, taps=taps)
        plans.append(p)
        xs.append(torch.from_numpy(_input(rng, "u8", C, T)).cuda())
        outs.append(torch.zeros((D, T - p.d_max), dtype=torch.int32, device="cuda"))
        want.append(p.dedisperse(xs[-1], nsamp=T))
    batch = dd.Batch(plans)
    batch.bind(xs, outs)
    batch.dedisperse()
    torch.cuda.synchronize()
    for p, x, o, w in zip(plans, xs, outs, want):
        assert torch.equal(o, w)
        assert torch.equal(p.dedisperse(x, nsamp=T), w)
        assert p.device_status() == 0

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

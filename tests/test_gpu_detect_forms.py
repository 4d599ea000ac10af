"""Detection stage and small tap launches at the edges of their branches: width lists of every
form, series at any 4-byte alignment, ties, normaliser channels of mixed weight runs, channel
statistics split over a cluster, and one CTA per pair of trials."""
import numpy as np
import pytest

import oracle
from oracle import ref

pytestmark = pytest.mark.gpu

OCTAVE = [1 << k for k in range(10)]
CHUNK = 256 * 31  # starts per chunk of a width list


@pytest.fixture(scope="module")
def dd():
    import torch
    from paper_1301_3968_gb300 import build
    build.build()
    import paper_1301_3968_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("mis", [0, 1, 3])
@pytest.mark.parametrize("seed,t_len,widths", [
    (1, 40, [1, 40]),                              # one segment; one start
    (2, CHUNK, OCTAVE),                            # the last start of a chunk
    (3, CHUNK + 1, OCTAVE),                        # the first of the next
    (4, 2 * CHUNK + 30, [31, 32, 34, 700]),        # tails shorter than a segment
    (5, 9001, list(range(1, 100, 3)) + [4096]),    # several groups, the widest list
    (6, 9001, [3, 4097]),                          # one past it: running sums
    (7, 9001, list(range(1, 100))),                # contiguous: sums from prefix sums
    (8, 9001, list(range(60, 80))),
])
def test_width_lists_on_integer_series(dd, seed, t_len, widths, mis):
    """Integer sums are exact, so the earliest start of the maximum is the oracle's; samples of
    0 and 1 give many ties.  S/N: fp32 mean and deviation, 1e-5."""
    import torch
    rng = np.random.default_rng(seed)
    C, D = 6, 5
    taps = rng.integers(1, 5, size=(D, C)).astype(np.int32)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, 100, "u8"), np.zeros(D))
    plan.set_profiles(delay=np.zeros((D, C), np.int32), taps=taps)
    ld = (t_len + mis + 3) // 4 * 4
    X = np.full((D, ld), 1 << 20, np.int32)        # (outside the series)
    X[:, mis:mis + t_len] = rng.integers(0, 2, size=(D, t_len))
    X[1, mis:mis + t_len] = 1                      # every start is a maximum
    X[2, mis:mis + t_len] = rng.integers(0, 1500, size=t_len)
    mu_c, sd_c = rng.uniform(0.0, 0.1, C), rng.uniform(0.5, 1.5, C)
    x = torch.from_numpy(X).cuda()[:, mis:]
    wl = np.array(widths, np.int32)
    peak, arg, _ = plan.boxcar_snr(x, wl, torch.from_numpy(mu_c).cuda(), torch.from_numpy(sd_c).cuda(),
                                   t_len=t_len)
    assert plan.device_status() == 0
    mu, sdw = ref.boxcar_norm(taps, wl, mu_c, sd_c)
    opeak, oarg, _ = ref.boxcar_snr(X[:, mis:mis + t_len].astype(np.int64), wl, mu, sdw)
    np.testing.assert_array_equal(arg.cpu().numpy(), oarg)
    np.testing.assert_allclose(peak.cpu().numpy(), opeak, rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("seed,C,nw,kmax", [
    (11, 1, 1, 8), (12, 255, 33, 8), (13, 257, 40, 5), (14, 300, 32, 60),
])
def test_normaliser_of_mixed_weight_runs(dd, seed, C, nw, kmax):
    """Channels of one weight beside channels whose weights vary.  Deviation: some 30 roundings of
    positive terms, 2e-6; sums of up to 40 + 31 samples around the mean add 1e-4 to the S/N."""
    import torch
    rng = np.random.default_rng(seed)
    D, T = 4, 600
    taps = rng.integers(1, kmax + 1, size=(D, C)).astype(np.int32)
    w = rng.uniform(0.5, 1.5, size=(D, C, kmax)).astype(np.float32)
    same = rng.random((D, C)) < 0.5
    same[0] = True
    w[same] = w[same][:, :1]
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "f32"), np.zeros(D))
    plan.set_profiles(delay=np.zeros((D, C), np.int32), taps=taps, weights=w)
    wl = np.arange(1, nw + 1, dtype=np.int32)
    mu_c, sd_c = rng.uniform(-0.1, 0.1, C), rng.uniform(0.5, 1.5, C)
    mu, sdw = ref.boxcar_norm(taps, wl, mu_c, sd_c, w=w)
    X = (mu[:, :1] + sdw[:, :1] * rng.standard_normal((D, T))).astype(np.float32)
    peak, _, _ = plan.boxcar_snr(torch.from_numpy(X).cuda(), wl, torch.from_numpy(mu_c).cuda(),
                                 torch.from_numpy(sd_c).cuda())
    opeak, _, _ = ref.boxcar_snr(X.astype(np.float64), wl, mu, sdw)
    np.testing.assert_allclose(peak.cpu().numpy(), opeak, rtol=1e-5, atol=1e-4)


@pytest.mark.parametrize("kind", ["u8", "f32"])
@pytest.mark.parametrize("seed,C,t_off,n", [
    (21, 1, 1, 1), (22, 2, 3, 17), (23, 3, 15, 4097), (24, 2, 5, 200003), (25, 700, 1, 5000), (26, 5, 0, 8192),
])
def test_channel_statistics_splits(dd, kind, seed, C, t_off, n):
    """uint8 sums are exact (two double roundings left); fp32 sums carry their remainders."""
    import torch
    rng = np.random.default_rng(seed)
    ld = (t_off + n + 15) // 16 * 16
    if kind == "u8":
        I = rng.integers(0, 256, size=(C, ld)).astype(np.uint8)
        I[0] = 255
    else:
        I = (100 + rng.standard_normal((C, ld))).astype(np.float32)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, ld, kind), np.zeros(1))
    m, s = plan.channel_stats(torch.from_numpy(I).cuda(), t_offset=t_off, nsamp=n)
    seg = I[:, t_off:t_off + n].astype(np.float64)
    tol = 1e-12 if kind == "u8" else 1e-9
    np.testing.assert_allclose(m.cpu().numpy(), seg.mean(axis=1), rtol=tol)
    np.testing.assert_allclose(s.cpu().numpy(), seg.std(axis=1), rtol=1e-6, atol=1e-5)


@pytest.mark.parametrize("kind", ["f32", "u8"])
@pytest.mark.parametrize("seed,D,t_out,kmax", [
    (31, 1, 1, 1), (32, 2, 767, 15), (33, 3, 768, 16), (34, 5, 769, 17), (35, 16, 2000, 32), (36, 17, 865, 33),
])
def test_small_tap_launches(dd, kind, seed, D, t_out, kmax):
    """Weights of every trial's own (no shared rows), shifted pairs and an odd last trial; at most
    5 x 33 terms: 165 roundings of 2^-24 of the absolute sum."""
    import torch
    rng = np.random.default_rng(seed)
    C = 5
    delay = rng.integers(0, 30, size=(D, C)).astype(np.int32)
    taps = rng.integers(1, kmax + 1, size=(D, C)).astype(np.int32)
    taps[0, 0] = kmax
    w = rng.standard_normal((D, C, kmax)).astype(np.float32)
    T = t_out + int((delay + taps - 1).max())
    ld = (T + 18) // 16 * 16
    I = (rng.integers(0, 256, size=(C, ld)).astype(np.uint8) if kind == "u8"
         else rng.standard_normal((C, ld)).astype(np.float32))
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, kind), np.zeros(D))
    plan.set_profiles(delay=delay, taps=taps, weights=np.zeros_like(w))
    plan.set_weights(torch.from_numpy(w).cuda())
    got = plan.dedisperse(torch.from_numpy(I).cuda(), t_offset=2, nsamp=T).cpu().numpy()
    assert plan.device_status() == 0
    want = oracle.c_dedisperse(I, delay, taps, w=w, t_offset=2, nsamp=T)
    scale = oracle.c_abs_scale(I, delay, taps, w=w, t_offset=2, nsamp=T)
    assert got.shape == (D, t_out)
    assert (np.abs(got - want) <= 1e-5 * scale).all()

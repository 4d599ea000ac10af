"""What a plan keeps between calls, when other calls come between: weights on the device, tables
that captured graphs read, scratch, and the schedule that a caller set."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dd():
    import torch
    from paper_1301_3968_gb300 import build
    build.build()
    import paper_1301_3968_gb300 as m
    torch.cuda.set_device(0)
    return m


def _weighted_plan(dd, C=12, D=20, T=2000, K=5):
    import torch
    rng = np.random.default_rng(3)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, T, "f32"), np.linspace(0.0, 40.0, D))
    plan.set_profiles(taps=np.full((D, C), K, np.int32), weights=np.ones((D, C, K), np.float32))
    x = torch.from_numpy(rng.standard_normal((C, T)).astype(np.float32)).cuda()
    w = torch.from_numpy(rng.standard_normal((2, D, C, K)).astype(np.float32)).cuda()
    g = torch.from_numpy(rng.standard_normal((D, T - plan.d_max)).astype(np.float32)).cuda()
    return plan, x, w[0].contiguous(), w[1].contiguous(), g


@pytest.mark.parametrize("between", ["nothing", "schedule", "method", "autotune", "other", "replay"])
def test_backward_uses_the_weights_of_its_forward(dd, between):
    """Whatever is done to the plan between a forward and its backward, the gradients are those of
    the forward's weights: new tables (which hold the host's weights), another forward, or a graph
    that sets weights."""
    import torch
    plan, x, w, w2, g = _weighted_plan(dd)

    def forward():
        xi, wi = x.clone().requires_grad_(True), w.clone().requires_grad_(True)
        return xi, wi, dd.DDFunction.apply(xi, wi, plan)

    xi, wi, y = forward()
    y.backward(g)
    want = y.detach().clone(), xi.grad.clone(), wi.grad.clone()
    graph = torch.cuda.CUDAGraph()
    if between == "replay":
        plan.set_weights(w2)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            plan.set_weights(w2)
    xi, wi, y = forward()
    if between == "schedule":
        plan.set_schedule(2, 3)
    elif between == "method":
        plan.set_method("direct")
    elif between == "autotune":
        plan.autotune(x, torch.empty_like(y))
    elif between == "other":
        dd.DDFunction.apply(x, w2, plan)
    elif between == "replay":
        graph.replay()
    y.backward(g)
    assert plan.device_status() == 0
    for a, b in zip(want, (y.detach(), xi.grad, wi.grad)):
        assert torch.equal(a, b)


def test_graph_of_a_plan_outlives_batches_of_it(dd):
    """A graph captured from a plan replays after a batch of the plan was made, run and closed, and
    after the plan's own calls since; the batch follows new profiles of a plan."""
    import torch
    rng = np.random.default_rng(5)
    C, T, D = 336, 9000, 110
    plans = [dd.Plan(dd.Band(C, 1130.0, 1.0, 1.0, T, "u8"), np.linspace(0, 600, D)) for _ in range(5)]
    xs = [torch.from_numpy(rng.integers(0, 256, size=(C, T // 16 * 16 + 16)).astype(np.uint8)).cuda() for _ in plans]
    want = [p.dedisperse(x, nsamp=T) for p, x in zip(plans, xs)]
    out = torch.empty_like(want[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plans[0].dedisperse(xs[0], nsamp=T, out=out)
    ids = [p.weights_id() for p in plans]
    batch = dd.Batch(plans)
    outs = [torch.zeros_like(w) for w in want]
    batch.bind(xs, outs)
    batch.dedisperse()
    torch.cuda.synchronize()
    assert all(torch.equal(o, w) for o, w in zip(outs, want))
    assert torch.equal(plans[0].dedisperse(xs[0], nsamp=T), want[0])
    assert [p.weights_id() for p in plans] == ids and 0 not in ids   # no table was uploaded anew
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want[0])
    delay, taps = plans[1].tables()
    plans[1].set_profiles(delay=delay[::-1], taps=taps[::-1])
    batch.dedisperse()
    torch.cuda.synchronize()
    assert torch.equal(outs[1], want[1].flip(0)) and torch.equal(outs[0], want[0])
    assert all(p.device_status() == 0 for p in plans)
    batch.close()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want[0])


def _u8_plan(dd, C=24, D=60, T=6000, nsamp=None):
    import torch
    rng = np.random.default_rng(7)
    delay = np.cumsum(rng.integers(0, 3, size=(D, C)), axis=0).astype(np.int32)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, nsamp or T, "u8"), np.zeros(D))
    plan.set_profiles(delay=delay, taps=np.full((D, C), 2, np.int32))
    plan.set_method("direct")
    return plan, torch.from_numpy(rng.integers(0, 256, size=(C, (T + 15) // 16 * 16)).astype(np.uint8)).cuda()


def _want(plan, x, T):
    import oracle
    delay, taps = plan.tables()
    return oracle.c_dedisperse(x.cpu().numpy(), delay, taps, nsamp=T).astype(np.int32)


def test_plans_for_detection_take_no_prefix_scratch(dd):
    """Prefix sums get their scratch from the call that reads them: a plan whose series come from
    elsewhere, or whose sums a batch forms, has none."""
    import torch
    C, T, D = 336, 60000, 300
    x = torch.zeros((C, T), dtype=torch.uint8, device="cuda")
    plans = [dd.Plan(dd.Band(C, 1130.0, 1.0, 1.0, T, "u8"), np.linspace(0, 600, D)) for _ in range(9)]
    assert all(p.method == "direct" for p in plans)
    plans[0].channel_stats(x, nsamp=T)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for p in plans[1:]:
        p.channel_stats(x, nsamp=T)
    torch.cuda.synchronize()
    # tables of some 4 MB a plan; the prefix sums of a block are 81 MB
    assert before - torch.cuda.mem_get_info()[0] < 8 * 20e6


def test_first_dedispersion_of_a_direct_plan_in_a_capture(dd):
    """With its tables on the device, a direct plan's first dedispersion may be a captured one."""
    import torch
    plan, x = _u8_plan(dd)
    T = x.shape[1]
    plan.channel_stats(x)
    out = torch.zeros((plan.ndm, T - plan.d_max), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.dedisperse(x, out=out)
    graph.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), _want(plan, x, T))


@pytest.mark.parametrize("limit_cols", [0, 4000])
def test_direct_calls_of_growing_length(dd, limit_cols):
    """Calls longer than any before get more scratch, or go in pieces where there is no more; a
    graph of a short one replays as it was."""
    import torch
    T = 30000
    plan, x = _u8_plan(dd, T=T, nsamp=1000)
    assert plan.d_max + 2 * 1088 < 4000
    plan.test_set_scratch_limit(limit_cols * plan.band.nchan * 4)
    want = _want(plan, x, T)
    out = torch.zeros((plan.ndm, 600), dtype=torch.int32, device="cuda")
    short = plan.dedisperse(x, nsamp=plan.d_max + 600)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.dedisperse(x, nsamp=plan.d_max + 600, out=out)
    for t_out in (700, 3000, 3300, 9000, T - plan.d_max):
        got = plan.dedisperse(x, nsamp=plan.d_max + t_out)
        np.testing.assert_array_equal(got.cpu().numpy(), want[:, :t_out])
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, short)
    np.testing.assert_array_equal(short.cpu().numpy(), want[:, :600])
    assert plan.device_status() == 0


@pytest.mark.parametrize("nch", [0, 2])
def test_direct_plan_without_room_for_prefix_sums(dd, nch):
    """Where the device has no room for a direct plan's prefix sums, its taps are summed one by one:
    the same sums and maxima, from the plan, the fused call and a batch, and with the next profiles;
    with room again, the shared rows."""
    import torch
    T = 6000
    plan, x = _u8_plan(dd, T=T)
    if nch:
        plan.set_schedule(nch, 4)
    want = _want(plan, x, T)
    mean, sd = plan.channel_stats(x, nsamp=T)
    wl = np.arange(1, 20, dtype=np.int32)
    peak, arg, _ = plan.boxcar_snr(torch.from_numpy(want).cuda(), wl, mean, sd)
    for limit in (1, 0):
        plan.test_set_scratch_limit(limit)
        np.testing.assert_array_equal(plan.dedisperse(x, nsamp=T).cpu().numpy(), want)
        plan.test_set_fused_parts(3)
        p1, a1, _ = plan.dedisperse_boxcar(x, wl, mean, sd, nsamp=T)
        assert torch.equal(p1.view(torch.int32), peak.view(torch.int32)) and torch.equal(a1, arg)
        plan.set_method("direct" if limit else "auto")      # new tables
        out = torch.zeros((plan.ndm, want.shape[1]), dtype=torch.int32, device="cuda")
        batch = dd.Batch([plan])
        batch.bind([x], [out])
        batch.dedisperse()
        np.testing.assert_array_equal(out.cpu().numpy(), want)
        batch.close()
        assert plan.device_status() == 0
    plan, x = _u8_plan(dd, T=T)
    plan.test_set_scratch_limit(1)
    plan.dedisperse(x, nsamp=T)
    delay, taps = plan.tables()
    plan.set_profiles(delay=delay[::-1], taps=taps[::-1] + 1)
    np.testing.assert_array_equal(plan.dedisperse(x, nsamp=T).cpu().numpy(), _want(plan, x, T))


def test_weights_from_the_device_keep_a_set_schedule(dd):
    """A schedule that a caller set stays when weights from the device replace the host's."""
    plan, x, w, w2, g = _weighted_plan(dd, D=60)
    assert plan.schedule()["trials_per_cta"] in (24, 48)      # rows: all trials have one weight
    plan.set_schedule(2, 3)
    plan.dedisperse(x)
    plan.set_weights(w)
    s = plan.schedule()
    assert (s["nch"], s["cs"], s["trials_per_cta"]) == (2, 3, 8)
    assert plan.device_status() == 0


@pytest.mark.parametrize("K", [1, 5, 16, 40])
@pytest.mark.parametrize("D", [1, 7, 33, 130])
def test_small_tap_launches_equal_the_full_one(dd, K, D):
    """A call that gives each pair unit a CTA returns the bits of a longer call of the same plan,
    which does not, at the edges of its tiles and of the trial blocks."""
    import torch
    rng = np.random.default_rng(K * 1000 + D)
    C, long = 5, 768 * (620 // ((D + 1) // 2) + 2)
    plan = dd.Plan(dd.Band(C, 1200.0, 1.0, 1.0, 4096, "f32"), np.zeros(D))
    delay = rng.integers(0, 60, size=(D, C)).astype(np.int32)
    plan.set_profiles(delay=delay, taps=np.full((D, C), K, np.int32), weights=np.ones((D, C, K), np.float32))
    plan.set_weights(torch.from_numpy(rng.standard_normal((D, C, K)).astype(np.float32)).cuda())
    n = long + plan.d_max
    x = torch.from_numpy(rng.standard_normal((C, (n + 3) // 4 * 4)).astype(np.float32)).cuda()
    want = plan.dedisperse(x, nsamp=n)
    for t in (1, 767, 768, 769, 2305):
        if t < long:
            assert torch.equal(plan.dedisperse(x, nsamp=t + plan.d_max), want[:, :t])
    assert plan.device_status() == 0

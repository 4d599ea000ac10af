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

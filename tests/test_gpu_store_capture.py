"""Captured calls of plans with a store, with eager calls in between: a graph keeps the store that it was captured on
when a later call takes a larger one."""
import time

import pytest

from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(prec, widths, points, mem_budget):
    from paper_2606_29702_gb300 import jet, specs
    plan = jet.Plan(specs.by_name("burgers", nu=0.01), widths, prec, store=True, mem_budget=mem_budget)
    p = torch.tensor(wl.pack(wl.xavier_layers(widths, 3, 0.1)), dtype=plan.dtype, device="cuda")
    xs = [torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], n, k), dtype=plan.dtype, device="cuda")
          for k, n in enumerate(points)]
    return plan, p, xs


def _capture(fn):
    g, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=stream):
        out = fn(stream)
    return g, out


def test_graph_keeps_its_store_when_the_plan_grows_one():
    plan, p, xs = _setup("bf16", [2, 256, 256, 256, 1], [3000, 9000, 20000], 2 << 30)
    want = [plan.backward(p, x)[0].clone() for x in xs[:1]]
    g, (grad, _, _) = _capture(lambda s: plan.backward(p, xs[0], stream=s))
    small = plan.info()["workspace_bytes"]
    plan.backward(p, xs[1])  # a larger store
    both = plan.info()["workspace_bytes"]
    for _ in range(2):
        grad.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(grad, want[0])
    del g
    torch.cuda.synchronize()
    time.sleep(0.5)  # the driver drops a graph's references on a thread of its own
    plan.backward(p, xs[2])  # the first store's graph is gone, and so is the second store
    assert both > small
    per_point = (both - small) / xs[1].shape[0]
    assert plan.info()["workspace_bytes"] <= small + 1.05 * per_point * (xs[2].shape[0] - xs[0].shape[0]) + (1 << 22)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_store_of_captured_and_eager_passes(prec):
    """A backward pass takes the jets of a forward pass that has run on its inputs, or computes its own: not those of a
    captured pass that has not run, and not what a replay put over an eager pass's."""
    widths = [2, 20, 20, 20, 1]
    plan, p, (x, y) = _setup(prec, widths, [700, 900], 1 << 28)
    want = [plan.backward(p, t)[0].clone() for t in (x, y)]
    tol = dict(rtol=0, atol=1e-5 * float(want[0].abs().max()))
    g, _ = _capture(lambda s: plan.forward(p, x, stream=s))
    assert torch.allclose(plan.backward(p, x)[0], want[0], **tol)  # the captured pass has not run
    plan.forward(p, y)
    g.replay()  # the graph's pass over the eager one's
    assert torch.allclose(plan.backward(p, y)[0], want[1], **tol)
    plan.forward(p, y)
    both, (grad, _, _) = _capture(lambda s: (plan.forward(p, x, stream=s), plan.backward(p, x, stream=s))[1])
    plan.forward(p, y)
    for _ in range(2):
        grad.zero_()
        both.replay()
        torch.cuda.synchronize()
        assert torch.allclose(grad, want[0], **tol)
    captured, (grad, _, _) = _capture(lambda s: plan.backward(p, y, stream=s))  # after an eager forward pass on y
    plan.forward(p, x)
    captured.replay()
    torch.cuda.synchronize()
    assert torch.allclose(grad, want[1], **tol)

"""Captured batched calls: a graph runs on the arguments it was captured with, and eager calls on theirs, in any order of
captures, replays and eager calls on one batch."""
import pytest

from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_captures_keep_their_arguments(prec):
    from paper_2606_29702_gb300 import jet, specs
    widths = [2] + [64] * 6 + [1]
    plans = [jet.Plan(specs.burgers(0.01), widths, prec) for _ in range(2)]
    ps = [torch.tensor(wl.pack(wl.xavier_layers(widths, 3 + k, 0.1)), dtype=torch.float32, device="cuda") for k in range(2)]
    sets = [[torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], n, k + n), dtype=torch.float32, device="cuda")
             for k, n in enumerate(points)] for points in ([700, 9000], [20000, 300], [129, 128])]
    b = jet.Batch(plans)
    stream = torch.cuda.Stream()

    def eager(i):
        grads, losses = b.backward(ps, sets[i])
        torch.cuda.synchronize()
        return torch.cat(grads + [losses]).clone()

    def capture(i):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            grads, losses = b.backward(ps, sets[i], stream=stream)
        return g, grads, losses

    def replay(c):
        for t in c[1] + [c[2]]:
            t.zero_()
        c[0].replay()
        torch.cuda.synchronize()
        return torch.cat(c[1] + [c[2]]).clone()

    want = [eager(0), eager(1), eager(2)]
    assert torch.equal(eager(0), want[0])
    c1 = capture(1)
    assert torch.equal(eager(1), want[1])  # the arguments of a capture that has not run
    c0 = capture(0)
    c2 = capture(2)
    assert torch.equal(replay(c1), want[1])
    assert torch.equal(eager(0), want[0])
    assert torch.equal(replay(c2), want[2])
    assert torch.equal(eager(0), want[0])
    assert torch.equal(replay(c0), want[0])
    assert torch.equal(replay(c1), want[1])
    assert torch.equal(eager(2), want[2])

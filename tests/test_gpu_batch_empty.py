"""Batched calls with members of no points: their gradient and loss are zero, as for a solo call, whatever earlier calls
left in the batch's buffers, and the other members are as without them.  21057 parameters are enough for FP32 sums per
chunk; the smaller network adds into FP64 slices."""
import pytest

from _common import rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,hidden", [("fp32", 6), ("fp32", 3), ("fp64", 3)])
def test_empty_members(prec, hidden):
    from paper_2606_29702_gb300 import jet, specs
    widths, points = [2] + [64] * hidden + [1], [900, 0, 30000, 0]
    plans = [jet.Plan(specs.burgers(0.01), widths, prec) for _ in points]
    dtype = plans[0].dtype
    ps = [torch.tensor(wl.pack(wl.xavier_layers(widths, 3 + k, 0.1)), dtype=dtype, device="cuda") for k in range(4)]
    full = [torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], 2000, k), dtype=dtype, device="cuda") for k in range(4)]
    xs = [torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], n, k), dtype=dtype, device="cuda").reshape(n, 2)
          for k, n in enumerate(points)]
    b = jet.Batch(plans)
    b.backward(ps, full)  # leaves sums in every member's buffers
    grads, losses = b.backward(ps, xs)
    for i, n in enumerate(points):
        if n == 0:
            assert not grads[i].any() and float(losses[i]) == 0.0
            continue
        g, loss, _ = plans[i].backward(ps[i], xs[i])
        assert rel_l2(grads[i].cpu().numpy(), g.cpu().numpy()) < 1e-6  # other chunks, FP32 sums
        assert abs(float(losses[i]) - float(loss)) <= 1e-12 * abs(float(loss))
    # every member empty: zero gradients, and a training step of zero moments moves nothing
    b.backward(ps, full)
    grads, losses = b.backward(ps, [x[:0] for x in full])
    assert not any(g.any() for g in grads) and not losses.any()
    before, ms, vs = [p.clone() for p in ps], [torch.zeros_like(p) for p in ps], [torch.zeros_like(p) for p in ps]
    b.train_step(ps, ms, vs, 1, 1e-3, [x[:0] for x in full])
    assert all(torch.equal(p, q) for p, q in zip(ps, before))

"""Chunk bounds of tensor-core batches: one member with more tiles than chunks, few members of unlike size, and enough
members for the least bound.  Tolerances: FP32 sums of a chunk's T tiles err by about T * 2^-24 relative (T < 10 here);
losses add up in FP64."""
import pytest

from _common import rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points", [[65537], [1], [40000, 129, 5000], [700 + 13 * i for i in range(39)]])
def test_batch_chunks_match_solo(points):
    from paper_2606_29702_gb300 import jet, specs
    widths = [2, 64, 64, 64, 1]
    ps = [torch.tensor(wl.pack(wl.xavier_layers(widths, 3 + k, 0.1)), dtype=torch.float32, device="cuda")
          for k in range(len(points))]
    xs = [torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], n, k), dtype=torch.float32, device="cuda")
          for k, n in enumerate(points)]
    plans = [jet.Plan(specs.burgers(0.01), widths, "bf16") for _ in points]
    solo = [p.backward(a, x) for p, a, x in zip(plans, ps, xs)]
    grads, losses = jet.Batch(plans).backward(ps, xs)
    torch.cuda.synchronize()
    for i in range(len(points)):
        assert rel_l2(grads[i].cpu().numpy(), solo[i][0].cpu().numpy()) < 1e-6
        assert abs(float(losses[i]) - float(solo[i][1])) <= 1e-12 * abs(float(solo[i][1]))

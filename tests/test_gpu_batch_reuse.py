"""Batches created one after another in a process: each uploads its own descriptors, whatever an earlier batch of the
same shapes and buffers left in recycled host memory."""
import numpy as np
import pytest

from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_batches_of_the_same_buffers(prec):
    from paper_2606_29702_gb300 import jet, specs
    widths = [2, 64, 64, 64, 1]
    ps = [torch.tensor(wl.pack(wl.xavier_layers(widths, 7 + k, 0.1)), dtype=torch.float32, device="cuda") for k in range(3)]
    xs = [torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], 300 + k, k), dtype=torch.float32, device="cuda") for k in range(3)]
    start = [p.clone() for p in ps]
    ms, vs = [torch.empty_like(p) for p in ps], [torch.empty_like(p) for p in ps]
    seen = []
    for _ in range(4):
        for p, p0, m, v in zip(ps, start, ms, vs):
            p.copy_(p0)
            m.zero_()
            v.zero_()
        batch = jet.Batch([jet.Plan(specs.burgers(0.01), widths, prec) for _ in range(3)])
        batch.train_step(ps, ms, vs, 1, 1e-3, xs)
        torch.cuda.synchronize()
        seen.append(torch.cat(ps).cpu().numpy())
        batch.close()
        del batch
    for p in seen[1:]:
        np.testing.assert_array_equal(p, seen[0])
    assert not np.array_equal(seen[0], torch.cat(start).cpu().numpy())

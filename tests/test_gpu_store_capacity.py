"""Capacity of the z-jet store: the points that the budget holds in groups of 4 * floor(256 / width) points (FP64: 2 *
floor(256 / width)), however many a tile takes, and passes on as many points as it says."""
import numpy as np
import pytest

from _common import rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,width,hidden", [("fp32", 64, 2), ("fp32", 128, 2), ("fp32", 64, 6), ("fp32", 20, 3), ("fp64", 64, 2),
                                               ("fp64", 20, 3), ("fp64", 100, 2)])
@pytest.mark.parametrize("groups", [1, 5])
def test_capacity(prec, width, hidden, groups):
    from paper_2606_29702_gb300 import jet, specs
    sp, widths = specs.burgers(0.01), [2] + [width] * hidden + [1]
    group = (2 if prec == "fp64" else 4) * (256 // width)
    n, point = groups * group, 4 * width * hidden * (8 if prec == "fp64" else 4)  # four channels
    plan = jet.Plan(sp, widths, prec, store=True, mem_budget=n * point)
    assert plan.info()["store_max_points"] >= n
    p = torch.tensor(wl.pack(wl.xavier_layers(widths, 3, 0.1)), dtype=plan.dtype, device="cuda")
    for points in (1, n - 1, n, n + 1):
        x = torch.tensor(wl.points([(-1.0, 1.0), (0.0, 1.0)], max(points, 1), 5), dtype=plan.dtype, device="cuda")
        want, loss, r = jet.Plan(sp, widths, prec).backward(p, x, want_r=True)
        r1, loss1 = plan.forward(p, x)
        g, loss2, _ = plan.backward(p, x)
        tol = 1e-13 if prec == "fp64" else 1e-6  # other tiles: sums in another order
        np.testing.assert_allclose(r1.cpu().numpy(), r.cpu().numpy(), rtol=0, atol=tol * float(r.abs().max()))
        assert rel_l2(g.cpu().numpy(), want.cpu().numpy()) <= tol
        assert abs(float(loss1) - float(loss)) <= 1e-12 * float(loss) and float(loss2) == pytest.approx(float(loss), rel=1e-12)

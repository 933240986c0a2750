"""Tensor-core calls that take a smaller tile than the plan's because their points do not fill the GPU: residual and
gradient against the same plan's largest tile (a tile override), at point counts around the tiles' edges.  The forward
arithmetic of a point does not depend on its tile, so residuals are equal bit by bit; gradients differ by the grouping of
FP32 sums over at most 64 points per sum (64 * 2^-24 = 3.8e-6 of their magnitudes, bound 2e-5)."""
import numpy as np
import pytest

from _common import rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [("burgers", 32, "bf16"), ("burgers", 64, "bf16"), ("allen_cahn", 128, "bf16"), ("ks", 64, "bf16"),
         ("ks", 64, "bf16x3"), ("ns_uvp", 32, "bf16"), ("ns_uvp", 64, "bf16"), ("ns_psi", 128, "bf16")]


@pytest.mark.parametrize("N", [1, 17, 1000, 4865, 9729, 20001])
@pytest.mark.parametrize("fam,width,prec", CASES, ids=["%s-%d-%s" % c for c in CASES])
def test_call_tile_matches_largest(fam, width, prec, N):
    from paper_2606_29702_gb300 import jet, specs
    sp = specs.by_name(fam, **specs.FAMILY_DEFAULTS[fam])
    widths = [sp.d_in] + [width] * 4 + [sp.n_out]
    plan = jet.Plan(sp, widths, prec)
    fixed = jet.Plan(sp, widths, prec, tile=plan.info()["tile_points"])
    p = torch.tensor(wl.pack(wl.xavier_layers(widths, 3, 0.1)), dtype=torch.float32, device="cuda")
    x = torch.tensor(wl.points([(0.0, 1.0)] * sp.d_in, N, 5), dtype=torch.float32, device="cuda")
    g, loss, r = plan.backward(p, x, want_r=True)
    g0, loss0, r0 = fixed.backward(p, x, want_r=True)
    np.testing.assert_array_equal(r.cpu().numpy(), r0.cpu().numpy())
    assert abs(float(loss) - float(loss0)) <= 1e-12 * abs(float(loss0))
    assert rel_l2(g.cpu().numpy(), g0.cpu().numpy()) <= 2e-5

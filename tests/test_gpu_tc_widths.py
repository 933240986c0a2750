"""Tensor-core form at every hidden width it accepts: multiples of 32 whose last 64-column chunk of the weights, or last
128-column block of a weight gradient, is narrower than the others.  Bound: the 6e-2 relative L2 of the BF16 parity
tests on stand-in shapes."""
import pytest

from _common import case, reference, rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", [False, True])
@pytest.mark.parametrize("width", [32, 64, 96, 128, 160, 192, 224, 256])
def test_every_width(width, store):
    from paper_2606_29702_gb300 import jet, specs
    spec, X, layers, src = case("burgers_2x20x4", 200, widths=[2, width, width, width, 1])
    L, r_ref, g_ref = reference(spec, X, layers)
    kw = dict(store=True, mem_budget=1 << 30) if store else {}
    plan = jet.Plan(specs.by_name(spec["family"], **spec["coefs"]), spec["widths"], "bf16", **kw)
    p = torch.tensor(wl.pack(layers), dtype=torch.float32, device="cuda")
    x = torch.tensor(X, dtype=torch.float32, device="cuda")
    g, loss, r = plan.backward(p, x, want_r=True)
    assert rel_l2(r.cpu().numpy(), r_ref) <= 6e-2
    assert rel_l2(g.cpu().numpy(), g_ref) <= 6e-2

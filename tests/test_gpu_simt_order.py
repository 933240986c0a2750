"""Order of the sums of an FP32 SIMT gradient: every element of a chunk's sums takes the groups of points one after
another, however many groups a tile holds.  All points share one position, and the sources make the groups' sums A, small,
small, -A: A drops out exactly, and what the small ones lose beside it depends on the order, far above the last FP32 bit
(A = 1e12 times the small ones: 2^-53 * 1e12 = 1e-4).  A plan with a z-jet store takes tiles of one group."""
import numpy as np
import pytest

from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [("value", [2] + [64] * 6 + [1]), ("value", [2] + [128] * 3 + [1]), ("value", [2, 136, 136, 136, 1]),
         ("value", [2, 96, 96, 96, 96, 3]), ("helmholtz", [3, 256, 256, 1]), ("helmholtz", [3, 64, 64, 64, 64, 64, 64, 1])]


@pytest.mark.parametrize("name,widths", CASES, ids=["-".join(map(str, w)) for _, w in CASES])
def test_groups_are_added_in_order(name, widths):
    from paper_2606_29702_gb300 import jet, specs
    if name == "value":  # residuals u_o - source_o
        spec = specs.Spec("value", 2, widths[-1], [[(1.0, [(o, (0, 0))])] for o in range(widths[-1])], has_source=True)
    else:
        spec = specs.helmholtz(2.0)
    group = 4 * (256 // max(widths))
    n = 304 * 8 * group  # whole patterns in every chunk
    rng = np.random.default_rng(5)
    big = rng.uniform(1e12, 2e12, (n // group // 4, 1))
    small = rng.normal(size=(n // group // 4, 2))
    f = np.concatenate([big, small, -big], axis=1).reshape(-1, 1, 1)
    src = np.broadcast_to(f, (n // group, group, spec.n_res)).reshape(n, spec.n_res)
    plan = jet.Plan(spec, widths, "fp32")
    one = jet.Plan(spec, widths, "fp32", store=True, mem_budget=1 << 32)
    assert plan.info()["wgrad_chunk_fp32"] == 1
    p = torch.tensor(wl.pack(wl.xavier_layers(widths, 3, 0.1)), dtype=torch.float32, device="cuda")
    x = torch.full((n, spec.d_in), 0.3, device="cuda")
    s = torch.tensor(np.ascontiguousarray(src), dtype=torch.float32, device="cuda")
    want, _, _ = one.backward(p, x, s)
    assert torch.isfinite(want).all()
    for _ in range(3):
        g, _, _ = plan.backward(p, x, s)
        np.testing.assert_array_equal(g.cpu().numpy(), want.cpu().numpy())

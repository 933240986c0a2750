"""A failed allocation is reported by the call's status alone: it stays no error of the CUDA runtime that the caller's
next check finds, and the caller can go on."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_out_of_memory_leaves_no_error_behind(prec):
    from paper_2606_29702_gb300 import jet, specs
    sp, widths = specs.burgers(0.01), [2, 64, 64, 1]
    with pytest.raises(jet.JetError) as err:
        jet.Plan(sp, widths, prec, store=True, mem_budget=1 << 46)
    assert err.value.status == 4  # JET_ERR_OOM
    x = torch.rand(100, 2, device="cuda", dtype=torch.float64 if prec == "fp64" else torch.float32)
    torch.cuda.synchronize()
    plan = jet.Plan(sp, widths, prec)
    p = torch.full((plan.info()["n_params"],), 0.1, device="cuda", dtype=plan.dtype)
    _, loss = plan.forward(p, x)
    assert torch.isfinite(loss)

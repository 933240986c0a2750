"""Reports of bounded waits that gave up: the first code is the one that is kept, and batches report theirs as plans do."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_first_code_is_kept():
    from paper_2606_29702_gb300 import jet
    # the hook's kernel waits twice in vain, with different codes, as a call and its teardown do
    for budget in (1_000, 500_000):
        assert jet.debug_wait_timeout(budget) == 6  # JET_ERR_TIMEOUT: the code of the first wait


def test_batch_reports_a_timed_out_wait():
    from paper_2606_29702_gb300 import jet, specs
    widths = [2, 32, 32, 1]
    plans = [jet.Plan(specs.burgers(0.01), widths, "bf16") for _ in range(2)]
    ps = [torch.full((plans[0].info()["n_params"],), 0.1, device="cuda") for _ in plans]
    xs = [torch.rand(100, 2, device="cuda") for _ in plans]
    b = jet.Batch(plans)
    want, _ = b.backward(ps, xs)
    b.debug_timeout(64)
    before, ms, vs = [p.clone() for p in ps], [torch.zeros_like(p) for p in ps], [torch.zeros_like(p) for p in ps]
    with pytest.raises(jet.JetError) as err:
        b.train_step(ps, ms, vs, 1, 1e-3, xs)
    assert err.value.status == 6 and "64" in str(err.value)  # JET_ERR_TIMEOUT
    assert all(torch.equal(p, q) for p, q in zip(ps, before))  # nothing ran on it
    got, _ = b.backward(ps, xs)  # reported once
    assert all(torch.equal(g, w) for g, w in zip(got, want))
    simt = jet.Batch([jet.Plan(specs.burgers(0.01), widths, "fp32")])
    with pytest.raises(jet.JetError):
        simt.debug_timeout(64)  # no waits there

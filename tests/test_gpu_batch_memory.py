"""Device memory of SIMT batches: sized by a call's work list (three items per CTA, two CTAs per SM, and one per member),
not by the bound of every member's chunks, and a batch that finds little memory is created with 16 chunks per member."""
import pytest

from _common import rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GIB = 1 << 30


def _members(family, widths, n, points):
    from paper_2606_29702_gb300 import jet, specs
    sp = specs.by_name(family, **specs.FAMILY_DEFAULTS[family])
    plans = [jet.Plan(sp, widths, "fp32") for _ in range(n)]
    ps = [torch.tensor(wl.pack(wl.xavier_layers(widths, 3 + k, 0.1)), dtype=torch.float32, device="cuda") for k in range(n)]
    xs = [torch.tensor(wl.points([(0.0, 1.0)] * sp.d_in, points, k), dtype=torch.float32, device="cuda") for k in range(n)]
    ss = [specs.helmholtz_source(x.double().cpu().numpy()) for x in xs] if sp.has_source else None
    return plans, ps, xs, None if ss is None else [torch.tensor(s, dtype=torch.float32, device="cuda") for s in ss]


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("family,widths,n", [("helmholtz", [3] + [256] * 8 + [1], 9), ("burgers", [2] + [64] * 6 + [1], 64),
                                             ("ns_psi", [3] + [128] * 4 + [2], 3)])
def test_memory_follows_the_work_list(family, widths, n):
    from paper_2606_29702_gb300 import jet
    plans, _, _, _ = _members(family, widths, n, 8)
    params, channels = plans[0].info()["n_params"], plans[0].info()["n_channels"]
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    before = _free()
    b = jet.Batch(plans)
    used = before - _free()
    b.close()
    # chunk sums, a run's FP32 sums per CTA, weight copies, jets of a tile of at most 32 points, allocation granules
    assert used <= (3 * ctas + n) * 8 * params + ctas * 4 * params + n * 12 * params + \
        ctas * 4 * channels * 32 * sum(widths[1:-1]) + (64 << 20)


def test_batch_with_little_memory():
    from paper_2606_29702_gb300 import jet
    plans, ps, xs, ss = _members("helmholtz", [3] + [256] * 8 + [1], 9, 700)
    full = jet.Batch(plans)
    want, loss = full.backward(ps, xs, sources=ss)
    full.close()
    torch.cuda.empty_cache()
    fill = torch.empty(_free() - 2 * GIB, dtype=torch.uint8, device="cuda")
    try:
        b = jet.Batch(plans)  # 4 GB with the chunks it would take
    finally:
        del fill
        torch.cuda.empty_cache()
    grads, losses = b.backward(ps, xs, sources=ss)
    for g, g0 in zip(grads, want):
        assert rel_l2(g.cpu().numpy(), g0.cpu().numpy()) < 1e-6  # other chunks, FP32 sums
    assert torch.allclose(losses, loss, rtol=1e-12, atol=0.0)


def test_tensor_core_batch_accepts_any_larger_memory():
    """A batch that fits some amount of free memory fits every larger one, whichever bound of chunks it ends with."""
    from paper_2606_29702_gb300 import jet, specs
    plans = [jet.Plan(specs.helmholtz(), [3] + [256] * 8 + [1], "bf16") for _ in range(9)]
    torch.cuda.empty_cache()
    jet.Batch(plans).close()
    most = torch.empty(_free() - 2 * GIB, dtype=torch.uint8, device="cuda")
    fits = []
    for mb in range(200, 1700, 20):
        fill = torch.empty(_free() - mb * (1 << 20), dtype=torch.uint8, device="cuda")
        try:
            jet.Batch(plans).close()
            fits.append(True)
        except jet.JetError as e:
            assert e.status == 4  # JET_ERR_OOM
            fits.append(False)
        del fill
        torch.cuda.empty_cache()
    del most
    torch.cuda.empty_cache()
    assert fits == sorted(fits) and fits[-1]

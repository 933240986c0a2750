"""SIMT tiles against the FP64 oracle where their split can go wrong: widths that take 4 or 8 units per thread,
layers narrower than the CTA (weight-gradient items shared by lanes), unequal widths, the 512-thread CTA of 256-wide
layers, networks without a jet GEMM, and point counts around and far from whole tiles.  Tolerances as for every SIMT
parity test: FP64 1e-12 (residual) and 1e-10 (gradient), FP32 1e-5."""
import numpy as np
import pytest

from _common import case, reference, rel_l2
from paper_2606_29702_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-12, 1e-10), "fp32": (1e-5, 1e-5)}
CASES = [("burgers_2x20x4", [2, 64, 1]), ("burgers_2x20x4", [2, 12, 40, 8, 1]), ("burgers_2x20x4", [2, 32, 64, 32, 1]),
         ("ks_2x64x5", [2, 20, 20, 1]), ("ks_2x64x5", [2, 128, 16, 1]), ("ns_uvp_2x64x6", [2, 4, 36, 3]),
         ("helmholtz_3x256x8", [3, 256, 8, 256, 1]), ("helmholtz_3x256x8", [3, 252, 24, 1]),
         ("ns_psi_3x128x6", [3, 64, 40, 2]),
         ("burgers_2x20x4", [2] + [128] * 7 + [1])]  # enough parameters for a warp per 32 of them in the reduction


def _plan(jet, specs, spec, prec, tile=None):
    return jet.Plan(specs.by_name(spec["family"], **spec["coefs"]), spec["widths"], prec, tile=tile)


def _tensors(plan, X, layers, src):
    def t(a):
        return None if a is None else torch.tensor(a, dtype=plan.dtype, device="cuda")
    return t(wl.pack(layers)), t(X), t(src)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("name,widths", CASES, ids=["-".join(map(str, w)) for _, w in CASES])
@pytest.mark.parametrize("N,tile", [(1, None), (29, None), (1217, None), (37, 16)])
def test_simt_tiles_match_oracle(name, widths, N, tile, prec):
    from paper_2606_29702_gb300 import jet, specs
    spec, X, layers, src = case(name, N, widths=widths)
    L, r_ref, g_ref = reference(spec, X, layers)
    try:
        plan = _plan(jet, specs, spec, prec, tile)
    except jet.JetError:  # a tile override whose two jet buffers one SM cannot hold is refused
        base = _plan(jet, specs, spec, prec)
        elem = 8 if prec == "fp64" else 4
        assert tile is not None and 2 * max(widths) * base.info()["n_channels"] * tile * elem > 200 * 1024
        return
    p, x, s = _tensors(plan, X, layers, src)
    g, loss, r = plan.backward(p, x, s, want_r=True)
    tr, tg = TOL[prec]
    assert rel_l2(r.cpu().numpy(), r_ref) <= tr
    assert rel_l2(g.cpu().numpy(), g_ref) <= tg
    assert abs(float(loss) - L) <= tr * abs(L)


def test_simt_batch_of_unequal_widths():
    """Members that alone take 8 units per thread, or CTAs of 512, share a launch with one that takes 4."""
    from paper_2606_29702_gb300 import jet, specs
    plans, ps, xs, ss, refs = [], [], [], [], []
    for k, widths in enumerate(([3, 256, 256, 1], [3, 12, 20, 1], [3, 64, 64, 64, 1])):
        spec, X, layers, src = case("helmholtz_3x256x8", 61 + 90 * k, widths=widths, seed_shift=k)
        plans.append(_plan(jet, specs, spec, "fp32"))
        refs.append(reference(spec, X, layers))
        for lst, t in zip((ps, xs, ss), _tensors(plans[-1], X, layers, src)):
            lst.append(t)
    grads, losses = jet.Batch(plans).backward(ps, xs, sources=ss)
    for g, loss, (L, _, g_ref) in zip(grads, losses.tolist(), refs):
        assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["fp32"][1]
        assert abs(loss - L) <= TOL["fp32"][0] * abs(L)
        assert np.isfinite(loss)


@pytest.mark.parametrize("N", [2000, 100000])
def test_fp32_sums_of_short_and_long_chunks(N):
    """FP32 weight-gradient sums that the reduction reads (chunks of one run) and that a chunk adds to FP64 slices run
    by run (more than 64 tiles of 8 points per CTA): repeating 50 points leaves the mean loss and its gradient."""
    from paper_2606_29702_gb300 import jet, specs
    spec, X, layers, src = case("ns_psi_3x128x6", 50, widths=[3, 128, 128, 128, 128, 2])
    L, _, g_ref = reference(spec, X, layers)
    plan = _plan(jet, specs, spec, "fp32", tile=8)
    assert plan.info()["wgrad_chunk_fp32"] == 1
    p, x, _ = _tensors(plan, np.tile(X, (N // 50, 1)), layers, src)
    g, loss, _ = plan.backward(p, x)
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["fp32"][1]
    assert abs(float(loss) - L) <= TOL["fp32"][0] * abs(L)


@pytest.mark.parametrize("name,widths", [("helmholtz_3x256x8", [3, 256, 256, 256, 1]), ("ns_psi_3x128x6", [3, 128, 128, 128, 128, 2]),
                                         ("burgers_2x20x4", [2] + [64] * 7 + [1]), ("ks_2x64x5", [2, 32, 32, 32, 1])])
def test_fp32_gradient_does_not_depend_on_the_tile(name, widths):
    """A plan with a z-jet store takes tiles of one group of points where it keeps FP32 sums, another takes several:
    the FP32 sums, and with them the gradient, are the same bits.  Without FP32 sums the FP64 adds of equal tile sums
    differ in order, at 2^-53 a term: at most the last bit of an FP32 value (2^-24 = 6e-8)."""
    from paper_2606_29702_gb300 import jet, specs
    spec, X, layers, src = case(name, 6011, widths=widths)
    plan = _plan(jet, specs, spec, "fp32")
    stored = jet.Plan(specs.by_name(spec["family"], **spec["coefs"]), widths, "fp32", store=True, mem_budget=1 << 30)
    p, x, s = _tensors(plan, X, layers, src)
    g, loss, _ = plan.backward(p, x, s)
    g1, loss1, _ = stored.backward(p, x, s)
    if plan.info()["wgrad_chunk_fp32"]:
        np.testing.assert_array_equal(g.cpu().numpy(), g1.cpu().numpy())
    assert rel_l2(g.cpu().numpy(), g1.cpu().numpy()) <= 6e-8
    assert abs(float(loss) - float(loss1)) <= 1e-12 * abs(float(loss1))

"""FP64 plans keep two CTAs per SM (one of more registers left the FP64 pipe idle between phases: 2 to 11% of a call with
seven and more channels)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,widths", [("burgers", [2, 20, 20, 1]), ("ks", [2, 64, 64, 1]), ("helmholtz", [3, 256, 256, 1]),
                                         ("helmholtz", [3, 64, 64, 1]), ("ns_psi", [3, 64, 64, 2])])
def test_two_ctas_per_sm(name, widths):
    from paper_2606_29702_gb300 import jet, specs
    plan = jet.Plan(specs.by_name(name, **specs.FAMILY_DEFAULTS[name]), widths, "fp64")
    assert plan.info()["ctas_per_sm"] == 2

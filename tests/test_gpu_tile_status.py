"""Tile overrides that no SM can hold are refused with the documented status."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("tile", [64, 256, 2040])
def test_too_large_a_tile_is_unsupported(prec, tile):
    from paper_2606_29702_gb300 import jet, specs
    with pytest.raises(jet.JetError) as err:
        jet.Plan(specs.helmholtz(), [3, 256, 256, 1], prec, tile=tile)
    assert err.value.status == 3  # JET_ERR_UNSUPPORTED

"""Reports of bounded waits that gave up: the first code is the one that is kept."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_first_code_is_kept():
    from paper_2606_29702_gb300 import jet
    # the hook's kernel waits twice in vain, with different codes, as a call and its teardown do
    for budget in (1_000, 500_000):
        assert jet.debug_wait_timeout(budget) == 6  # JET_ERR_TIMEOUT: the code of the first wait

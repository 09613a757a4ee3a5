"""CPU test of what a run makes of the device's error word: one rule for plain,
recorded, batched and allocation-free runs. A wait that ran out (of a bulk copy
or of a flow launch's tile) is STEPS_ERR_TIMEOUT and closes the simulations,
whatever else the word says; the other bits are STEPS_ERR_STATE."""
import pytest


@pytest.fixture(scope="module")
def capi():
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi as c
    return c


@pytest.mark.parametrize("word,code,closed,text", [
    (0, 0, False, None), (1, -7, False, "negative count"), (2, -7, False, "2^24 reactions"),
    (3, -7, False, "2^24 reactions"), (4, -6, True, "bulk copy"), (8, -6, True, "flow launch"),
    (9, -6, True, "flow launch"), (12, -6, True, "bulk copy")])
def test_error_word(capi, word, code, closed, text):
    assert capi.steps_debug_error_word(word) == (code, closed)
    if text:
        assert text in capi.lib.steps_last_error().decode()

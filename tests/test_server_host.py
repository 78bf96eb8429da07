"""Host-side checks of the solve server (no GPU needed)."""
import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_1304_5546_gb300 import build as B
    B.build()
    from paper_1304_5546_gb300 import _lib
    return _lib


# CUDA error codes: success, not ready, illegal address, launch failure,
# out of memory, context destroyed, unknown
@pytest.mark.parametrize("code,state", [(0, "DONE"), (600, "RUNNING"), (700, "FAILED"),
                                        (719, "FAILED"), (2, "FAILED"), (709, "FAILED"),
                                        (999, "FAILED")])
def test_state_of_a_result_by_its_event(lib, code, state):
    assert lib.load().dg_test_result_state(code) == getattr(lib, "DG_REQUEST_" + state)

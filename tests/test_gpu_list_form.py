"""The GPU tests of the list form at small sizes, with the form taken whatever the
mesh size (by rule it is kept for large meshes)."""
import pytest

from test_gpu_list import *  # noqa: F401,F403
from test_gpu_list import capi as _capi, pytestmark  # noqa: F401


@pytest.fixture(autouse=True)
def _form(capi):  # noqa: F811
    capi.steps_debug_form(2)
    yield
    capi.steps_debug_form(0)

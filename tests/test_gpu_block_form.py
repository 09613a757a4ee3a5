"""GPU parity of block tiles compiled for models of 13 or more species, taken for
every window here (by rule they run large meshes at few molecules per tet): the
tests of the list form and of dense states of many species, in their launch
forms, batches, recordings and leave laws."""
import pytest

from test_gpu_list import *  # noqa: F401,F403
from test_gpu_list import capi as _capi, pytestmark  # noqa: F401
from test_gpu_many_species import test_dense_states, test_full_word_streams  # noqa: F401


@pytest.fixture(autouse=True)
def _form(capi):  # noqa: F811
    capi.steps_debug_form(3)
    yield
    capi.steps_debug_form(0)

"""GPU test of the bounded wait of warp tiles in flow launches: a warp waits for
its own tile and those of its face neighbours; whichever has not finished, the
wait gives up after its cycle limit with an error status, and the device stays
usable."""
import numpy as np
import pytest

import oracle
from paper_1610_02258_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi as c
    return c


def test_neighbour_wait_completes_and_times_out(capi):
    capi.steps_debug_flow_nbr_wait(-1, 1 << 24)
    for late in (0, 1, 2, 31, 39):  # 1: its own tile
        for limit in (1 << 12, 1 << 20):
            with pytest.raises(capi.StepsError) as e:
                capi.steps_debug_flow_nbr_wait(late, limit)
            assert e.value.code == -6 and "did not complete" in str(e.value)
    for late, limit in ((40, 1 << 12), (-2, 1 << 12), (0, 0), (0, (1 << 31) + 1)):
        with pytest.raises(capi.StepsError) as e:
            capi.steps_debug_flow_nbr_wait(late, limit)
        assert e.value.code == -1
    w = I.config2(nx=4, t_end=1e-3)
    g = capi.from_workload(w, specialize=1, flow=True)
    g.run(w.t_end)
    o = oracle.from_workload(w, prec=32)
    o.run(w.t_end)
    assert np.array_equal(g.get_counts(), o.get_counts())

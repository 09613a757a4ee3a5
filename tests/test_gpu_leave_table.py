"""The EXP leave law's tables (device, with the entries near an integer decided
by the host) against the oracle's thresholds, every entry equal: windows of
tau, of most of it and of almost none, species over eight decades of diffusion
constant and an immobile one, enough entries that the host decides some."""
import numpy as np
import pytest

import oracle
from paper_1610_02258_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [1, 40])
def test_leave_table_equals_the_oracle(nx):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi
    h = 0.6 * I.UM
    verts, tets = I.kuhn_box_mesh(nx, 17, 17, h)
    verts = I.jitter_box_vertices(verts, h, 0.2, seed=1)
    diff = [1e-11, 9.99e-12, 4.3e-12, 1e-12, 2e-13, 1e-14, 1e-16, 1e-19, 0.0]
    m = I.model_from_lists([f"S{i}" for i in range(9)], diff, [])
    g = capi.Simulation(verts, tets, m, 1, leave_law=capi.STEPS_LEAVE_EXP)
    o = oracle.OracleSim(verts, tets, m, seed=1, prec=32, leave=oracle.EXP)
    assert g.tau == o.tau
    decided = 0
    for f in (1.0, 0.83, 0.31, 1e-3, 1e-9):
        got, n = capi.steps_debug_leave_table(g._sim, f * g.tau, 9, g.nt)
        decided += n
        for s in range(9):
            assert np.array_equal(got[s], o.species_thresholds(s, f * o.tau)[0][:, 3]), (f, s)
    if nx > 1:  # 69,360 tets: 1.5 million mobile entries with a product above 1, one in 2^15
        assert 10 < decided < 200

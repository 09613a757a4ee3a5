"""GPU parity of the EXP leave law on either side of the table size up to which
the host computes a shortened window's table (8,192 entries: 8 species of 1,020
and 1,026 tets): runs, recordings and a batch whose runs end off the window
grid at a different length each time, against the oracle, bit for bit."""
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


def _pair(capi, cells, seed=2):
    names = [f"S{i}" for i in range(8)]
    m = I.model_from_lists(names, [1e-11 * 0.4 ** i for i in range(7)] + [0.0],
                           [([names[0]], [names[7]], 100.0), ([names[7]], [names[1]], 50.0)])
    verts, tets = I.kuhn_box_mesh(cells, 1, 1, 0.5 * I.UM)
    c = np.random.default_rng(cells).integers(0, 20, (8, tets.shape[0])).astype(np.int32)
    g = capi.Simulation(verts, tets, m, seed, leave_law=capi.STEPS_LEAVE_EXP)
    o = oracle.OracleSim(verts, tets, m, seed=seed, occ=oracle.OCC, prec=32, leave=oracle.EXP)
    for obj in (g, o):
        obj.set_counts(c)
    return g, o


@pytest.mark.parametrize("cells", [1, 170, 171])
def test_runs_and_recordings(capi, cells):
    import torch
    g, o = _pair(capi, cells)
    for w in (2.3, 0.4, 17.9):
        t = o.time + w * o.tau
        g.run(t)
        o.run(t)
        assert np.array_equal(g.get_counts(), o.get_counts())
    dt, t0 = 1.7 * o.tau, o.time
    tets = np.arange(g.nt, dtype=np.int32)
    buf = torch.zeros((12, 8, g.nt), dtype=torch.int32, device="cuda")
    assert g.run_record(t0 + 12.5 * dt, dt, np.arange(8, dtype=np.int32), tets, buf.data_ptr(), 12) == 12
    for k in range(12):
        o.run(t0 + (k + 1) * dt)
        assert np.array_equal(buf[k].cpu().numpy(), o.get_counts())


def test_batch_of_both_sizes(capi):
    pairs = [_pair(capi, cells, 3 + cells) for cells in (170, 171, 40)]
    b = capi.Batch([g for g, _ in pairs], block=256)
    for w in (2.3, 5.6):
        ends = [o.time + (w + 0.1 * j) * o.tau for j, (_, o) in enumerate(pairs)]
        b.run(ends)
        for (g, o), t in zip(pairs, ends):
            o.run(t)
            assert g.windows == o.windows and np.array_equal(g.get_counts(), o.get_counts())
    b.close()

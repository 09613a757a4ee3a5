"""The check of the counts a caller hands in, where its loads have edges: one
negative count first, in the middle or last among 6 to 3,078 (not always
whole groups of four), and device counts that start off a 16-byte boundary."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("S,cells", [(1, 1), (1, 57), (3, 171)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_a_negative_count_is_found(capi, S, cells, offset):
    import torch
    verts, tets = I.kuhn_box_mesh(cells, 1, 1, 0.5 * I.UM)
    nt = tets.shape[0]
    m = I.model_from_lists([f"S{i}" for i in range(S)], [1e-12] * S, [])
    sim = capi.Simulation(verts, tets, m, 7, specialize=-1)
    good = np.arange(S * nt, dtype=np.int32).reshape(S, nt)
    sim.set_counts(good)
    n = S * nt
    for at in {0, 1, n // 2, n - 2, n - 1}:
        bad = good.copy()
        bad.reshape(-1)[at] = -5
        with pytest.raises(Exception):
            sim.set_counts(bad)
        assert np.array_equal(sim.get_counts(), good)
        buf = torch.zeros(n + 4, dtype=torch.int32, device="cuda")
        view = buf[offset:offset + n]
        view.copy_(torch.from_numpy(bad.reshape(-1)))
        torch.cuda.synchronize()
        with pytest.raises(Exception):
            capi.steps_run_noalloc(sim._sim, view.data_ptr(), sim.time + sim.tau)
        assert np.array_equal(view.cpu().numpy(), bad.reshape(-1)) and sim.time == 0.0
    sim.close()

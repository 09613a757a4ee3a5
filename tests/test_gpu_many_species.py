"""GPU parity of the warp tiles compiled for models of 13 to 32 species in dense
states (above the density of the list form) against the CPU oracle, bit for
bit: the wider tables of words per species (a third row from 29 species on, no
padding row at 16, 20, 28 and 32), full word streams that the table holds and
longer ones, both launch forms, both leave laws."""
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


def _model(S):
    names = [f"S{i}" for i in range(S)]
    diff = [1e-11 / (1 + i % 7) for i in range(S)]
    diff[5] = 0.0
    reac = [([], [names[0]], 1e-5), ([names[0]], [names[1]], 100.0), ([names[1], names[2]], [names[S - 1]], 1e6),
            ([names[4], names[4]], [names[5]], 1e6), ([names[S - 1]], [names[2], names[3]], 50.0)]
    return I.model_from_lists(names, diff, reac)


def _check(capi, S, values, leave=0, flow=None, block=256):
    verts, tets = I.kuhn_box_mesh(5, 3, 3, 0.5 * I.UM)
    nt = tets.shape[0]
    m = _model(S)
    counts = np.random.default_rng(S).choice(np.asarray(values, np.int32), size=(S, nt)).astype(np.int32)
    assert np.count_nonzero(counts) > nt  # dense: not the list form
    g = capi.Simulation(verts, tets, m, 13, specialize=1, leave_law=leave, flow=flow, block=block)
    o = oracle.OracleSim(verts, tets, m, seed=13, occ=oracle.OCC, prec=32, leave=leave)
    for obj in (g, o):
        obj.set_counts(counts)
    for k in (2.0, 4.6):
        g.run(k * o.tau)
        o.run(k * o.tau)
        assert np.array_equal(g.get_counts(), o.get_counts())
    assert g.specialized and o.events > 0


@pytest.mark.parametrize("S", [14, 16, 17, 20, 28, 29, 31, 32])
@pytest.mark.parametrize("flow", [False, True])
def test_dense_states(capi, S, flow):
    _check(capi, S, [0, 0, 1, 2, 5, 15, 16, 33], flow=flow)


@pytest.mark.parametrize("S", [16, 20, 28, 32])
@pytest.mark.parametrize("leave", [0, 1])
def test_full_word_streams(capi, S, leave):
    """Tets of up to 127 words, then of up to 480."""
    _check(capi, S, [0, 1, 127 // S], leave=leave, flow=leave == 0)
    _check(capi, S, [9, 13, 14, 15], leave=leave, block=64 if leave else 512)

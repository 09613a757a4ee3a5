"""GPU tests of when a run takes the list form (models of 13 or more species in
sparse states; here without the rule's mesh size) and when the tiles, seen from whether a run's tuning of the
launch form took place (tiles) or not (list form), with counts equal to the
oracle's either way."""
import numpy as np
import pytest

import oracle
from paper_1610_02258_gb300 import inputs as I

pytestmark = pytest.mark.gpu

S = 14


@pytest.fixture
def capi(_capi):
    _capi.steps_debug_form(2)
    yield _capi
    _capi.steps_debug_form(0)


@pytest.fixture(scope="module")
def _capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi as c
    return c


def _pair(capi, seed, grid=(8, 6, 5), source=0.0):
    names = [f"S{i}" for i in range(S)]
    reac = [([names[0]], [names[1]], 30.0), ([names[1]], [names[0]], 20.0)]
    if source:
        reac.append(([], [names[2]], source))
    m = I.model_from_lists(names, [1e-11 / (1 + i) for i in range(S)], reac)
    verts, tets = I.kuhn_box_mesh(*grid, 0.5 * I.UM)
    g = capi.Simulation(verts, tets, m, seed, specialize=1)
    o = oracle.OracleSim(verts, tets, m, seed=seed, occ=oracle.OCC, prec=32)
    return g, o


def _run(g, o, windows=80.4):
    t = o.time + windows * o.tau
    g.run(t)
    o.run(t)
    assert g.windows == o.windows and np.array_equal(g.get_counts(), o.get_counts())


def _tiles(g):
    return g.flow[1][0] > 0.0


def _set(capi, g, o, c, species=None):
    o.set_counts(c)
    if species is None:
        g.set_counts(c)
    for s in species or []:
        capi.steps_set_counts(g._sim, s, c[s])


def test_empty_species_set_one_by_one_leave_a_dense_state_dense(capi):
    g, o = _pair(capi, 1)
    c = np.zeros((S, g.nt), np.int32)
    c[0] = 9
    _set(capi, g, o, c)
    _set(capi, g, o, c, range(1, S))
    _run(g, o)
    assert _tiles(g)


def test_a_sparse_state_set_species_by_species_is_listed(capi):
    g, o = _pair(capi, 2)
    c = np.zeros((S, g.nt), np.int32)
    c[0] = 9
    _set(capi, g, o, c)
    c[0] = 0
    c[:, ::60] = 2
    _set(capi, g, o, c, range(S))
    _run(g, o)
    assert not _tiles(g)
    c = o.get_counts()
    c[3] = 5
    _set(capi, g, o, c, [3])
    _run(g, o)
    assert _tiles(g)



def _filling(capi, seed):
    """A few molecules, and a source in every tet that fills the mesh."""
    g, o = _pair(capi, seed, source=3e-5)
    c = np.zeros((S, g.nt), np.int32)
    c[0, ::60] = 2
    _set(capi, g, o, c)
    return g, o


def test_a_recording_leaves_the_list_form(capi):
    """Intervals too short for a look of their own (100 windows) add up to one."""
    import torch
    g, o = _filling(capi, 3)
    tets = np.arange(0, g.nt, 9, dtype=np.int32)
    buf = torch.zeros((15, 1, tets.size), dtype=torch.int32, device="cuda")
    dt = 100 * o.tau
    assert g.run_record(15 * dt, dt, np.array([2], np.int32), tets, buf.data_ptr(), 15) == 15
    assert _tiles(g)
    for k in range(15):
        o.run((k + 1) * dt)
        assert np.array_equal(buf[k].cpu().numpy(), o.get_counts()[[2]][:, tets])
    assert np.array_equal(g.get_counts(), o.get_counts())


def test_a_batch_run_leaves_the_list_form(capi):
    """One long run of a member that fills up and one that is dense from the start:
    three launches a window (tiles, list, advance) become two on the way."""
    pairs = [_filling(capi, 4), _pair(capi, 5, (6, 6, 5), 3e-5)]
    g, o = pairs[1]
    _set(capi, g, o, np.full((S, g.nt), 2, np.int32))
    b = capi.Batch([p[0] for p in pairs], block=256, specialize=1)
    windows = 1500.4
    b.run([windows * o.tau for _, o in pairs])
    for g, o in pairs:
        o.run(windows * o.tau, threads=8)
        assert g.windows == o.windows == 1501
        assert np.array_equal(g.get_counts(), o.get_counts())
    assert 1024 * 3 <= b.info[1] <= 1024 * 3 + 480 * 2
    b.close()


def test_a_new_batch_has_its_members_work_lists(capi):
    """The lists of a batch fit its members' states from its creation on: the first
    run of a sparse and a dense member allocates (and frees) nothing."""
    pairs = [_pair(capi, 6), _pair(capi, 7, (6, 6, 5))]
    for (g, o), every in zip(pairs, (60, 1)):
        c = np.zeros((S, g.nt), np.int32)
        c[:, ::every] = 2
        _set(capi, g, o, c)
    b = capi.Batch([p[0] for p in pairs], block=256, specialize=1)
    made = capi.steps_debug_fail_alloc(0)
    b.run([20.4 * o.tau for _, o in pairs])
    assert capi.steps_debug_fail_alloc(0) == made
    assert b.info[1] == 3 * 21
    for g, o in pairs:
        o.run(20.4 * o.tau)
        assert np.array_equal(g.get_counts(), o.get_counts())
    b.close()

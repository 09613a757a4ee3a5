"""Device allocations that fail (made to, on the host: steps_debug_fail_alloc)
leave simulations and batches as they were: the call reports STEPS_ERR_OOM, and
the same call afterwards runs to the oracle's counts."""
import numpy as np
import pytest

import oracle
from paper_1610_02258_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def _capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi as c
    return c


@pytest.fixture
def capi(_capi):
    _capi.steps_debug_form(2)  # the list form in sparse states of these small meshes
    yield _capi
    _capi.steps_debug_fail_alloc(0)
    _capi.steps_debug_form(0)


def _many_species():
    names = [f"S{i}" for i in range(14)]
    reac = [([names[0]], [names[1]], 300.0), ([names[1]], [names[2], names[3]], 200.0)]
    return I.model_from_lists(names, [1e-11 / (1 + i) for i in range(14)], reac)


def _members(capi, kind):
    """(simulations, oracles) of one model structure; `listed`: sparse and dense states of 14 species."""
    out = []
    for j, nx in enumerate((9, 6, 4)):
        if kind == "listed":
            verts, tets = I.kuhn_box_mesh(nx, 6, 5, 0.5 * I.UM)
            m = _many_species()
            c = np.random.default_rng(j).integers(0, 4, (14, tets.shape[0])).astype(np.int32)
            if j < 2:
                c[:, 20:] = 0  # sparse: the list form
            seed = 60 + j
        else:
            w = I.config2(seed=60 + j, nx=nx, ny=3, nz=3)
            verts, tets, m, c, seed = w.verts, w.tets, w.model, w.counts, w.seed
        g = capi.Simulation(verts, tets, m, seed, specialize=1)
        o = oracle.OracleSim(verts, tets, m, seed=seed, occ=oracle.OCC, prec=32)
        for obj in (g, o):
            obj.set_counts(c)
        out.append((g, o))
    return [p[0] for p in out], [p[1] for p in out]


@pytest.mark.parametrize("kind", ["box", "listed"])
@pytest.mark.parametrize("block,flow", [(256, False), (0, False), (256, True), (0, True)])
def test_batch_runs_after_a_failed_allocation(capi, kind, block, flow):
    """Each allocation of a first run in turn; the tuned block sizes (block 0)
    and the flow words are all allocated before the first window."""
    for nth in range(1, 20):
        sims, refs = _members(capi, kind)
        b = capi.Batch(sims, block=block, specialize=1, flow=flow)
        ends = [20.4 * o.tau for o in refs]
        capi.steps_debug_fail_alloc(nth)
        failed = False
        try:
            b.run(ends)
        except capi.StepsError as e:
            assert e.code == -4, e
            failed = True
            assert all(s.windows == 0 for s in sims)
        capi.steps_debug_fail_alloc(0)
        if failed:
            b.run(ends)
        for s, o, t in zip(sims, refs, ends):
            o.run(t)
            assert s.windows == o.windows and np.array_equal(s.get_counts(), o.get_counts()), nth
        b.close()
        if not failed:
            break
    else:
        raise AssertionError("a run makes more allocations than expected")


def _sparse(capi, **kw):
    verts, tets = I.kuhn_box_mesh(6, 6, 5, 0.5 * I.UM)
    m = _many_species()
    c = np.zeros((14, tets.shape[0]), np.int32)
    c[:4, ::20] = 5
    g = capi.Simulation(verts, tets, m, 70, specialize=1, **kw)
    o = oracle.OracleSim(verts, tets, m, seed=70, occ=oracle.OCC, prec=32)
    for obj in (g, o):
        obj.set_counts(c)
    return g, o, c


def _equal_run(g, o):
    g.run(20.4 * o.tau)
    o.run(20.4 * o.tau)
    assert g.windows == o.windows and np.array_equal(g.get_counts(), o.get_counts())


def _list_bytes(g):
    return (10 + g.S) * ((g.nt + 31) // 32 * 32) * 4 + 16


def test_a_simulation_needs_no_room_for_the_list_form(capi):
    """Each allocation of a creation in turn: those of the simulation proper end it,
    those of the list form (sparse states of 13 or more species) do not."""
    full = _sparse(capi)[0].device_bytes
    without = refused = 0
    for nth in range(1, 40):
        capi.steps_debug_fail_alloc(nth)
        try:
            g, o, _ = _sparse(capi)
        except capi.StepsError as e:
            assert e.code == -4 and without == 0, e
            refused += 1
            continue
        finally:
            capi.steps_debug_fail_alloc(0)
        if g.device_bytes == full:
            break
        assert g.device_bytes == full - _list_bytes(g)
        without += 1
        _equal_run(g, o)
    assert without >= 5 and refused >= 5


def test_a_clone_needs_no_room_for_the_list_form(capi):
    g, o, c = _sparse(capi)
    capi.steps_debug_fail_alloc(1)
    k = g.clone(70)
    assert k.device_bytes == g.device_bytes - _list_bytes(g)
    k.set_counts(c)
    _equal_run(k, o)


def test_flow_simulations_hold_no_list_buffers(capi):
    g, o, _ = _sparse(capi, flow=True)
    assert g.device_bytes == _sparse(capi)[0].device_bytes - _list_bytes(g)
    _equal_run(g, o)

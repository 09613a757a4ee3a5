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
    yield _capi
    _capi.steps_debug_fail_alloc(0)


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

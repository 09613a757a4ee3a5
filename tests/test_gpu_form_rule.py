"""GPU parity of the forms that the rule and the tuning choose for a compiled
model of 30 species on meshes just above a resident wave of warp tiles: sparse
and dense states of one simulation (each tuned for itself: window and flow
launches of warp tiles and of block tiles all run), short runs, and a batch
that is above a wave only together, against the oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_1610_02258_gb300 import inputs as I

pytestmark = pytest.mark.gpu

THREADS = max(1, min(32, os.cpu_count() or 1))
S = 30


@pytest.fixture(scope="module")
def capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi as c
    return c


def _pair(capi, nx, seed):
    names = [f"S{i}" for i in range(S)]
    reac = [([names[0]], [names[1]], 60.0), ([names[1], names[2]], [names[3]], 1e7), ([names[3]], [names[2], names[1]], 50.0)]
    m = I.model_from_lists(names, [1e-11 / (1 + i % 9) for i in range(S)], reac)
    verts, tets = I.kuhn_box_mesh(nx, 17, 17, 0.6 * I.UM)
    g = capi.Simulation(verts, tets, m, seed)
    o = oracle.OracleSim(verts, tets, m, seed=seed, occ=oracle.OCC, prec=32)
    return g, o


def _place(pair, per_tet, seed):
    g, o = pair
    rng = np.random.default_rng(seed)
    c = np.zeros((S, g.nt), np.int32)
    n = int(per_tet * g.nt)
    np.add.at(c, (rng.integers(0, S, n), rng.integers(0, g.nt, n)), 1)
    for obj in pair:
        obj.set_counts(c)


def _equal(g, o):
    assert g.windows == o.windows and np.array_equal(g.get_counts(), o.get_counts())


def test_tuned_forms_of_sparse_and_dense_states(capi):
    pair = g, o = _pair(capi, 47, 5)
    assert g.nt > 77824 and g.specialized
    for per_tet, windows in ((0.3, 4.4), (0.3, 93.4), (3.0, 92.0), (0.3, 3.3)):
        _place(pair, per_tet, int(10 * per_tet))
        t = o.time + windows * o.tau
        g.run(t)
        o.run(t, threads=THREADS)
        _equal(g, o)
    assert g.flow[1][0] > 0.0


def test_batch_above_a_wave_together(capi):
    pairs = [_pair(capi, 25, 6), _pair(capi, 24, 7)]
    for pair in pairs:
        _place(pair, 0.4, 3)
    b = capi.Batch([g for g, _ in pairs])
    for windows in (17.4, 3.2):
        ends = [o.time + windows * o.tau for _, o in pairs]
        b.run(ends)
        for (g, o), t in zip(pairs, ends):
            o.run(t, threads=THREADS)
            _equal(g, o)
    assert b.specialized
    b.close()


@pytest.mark.parametrize("per_tet", [0.3, 3.0])
def test_run_time_batches_on_either_side_of_the_density(capi, per_tet):
    """Members of 10 and 3 species on the kernels for models given at run time: block
    tiles below half a molecule per tet, warp tiles above; then the other way."""
    ws = [I.config2(seed=80, nx=3), I.config1(seed=81), I.config2(seed=82, nx=2)]
    sims, refs = [], []
    for w in ws:
        sims.append(capi.Simulation(w.verts, w.tets, w.model, w.seed, specialize=-1))
        refs.append(oracle.OracleSim(w.verts, w.tets, w.model, seed=w.seed, occ=oracle.OCC, prec=32))
    b = capi.Batch(sims, block=128, specialize=-1)
    for k, d in enumerate((per_tet, 3.3 - per_tet)):
        for g, o in zip(sims, refs):
            rng = np.random.default_rng(k)
            c = np.zeros((g.S, g.nt), np.int32)
            n = int(d * g.nt)
            np.add.at(c, (rng.integers(0, g.S, n), rng.integers(0, g.nt, n)), 1)
            g.set_counts(c)
            o.set_counts(c)
        ends = [o.time + 18.4 * o.tau for o in refs]
        b.run(ends)
        for g, o, t in zip(sims, refs, ends):
            o.run(t)
            _equal(g, o)
    b.close()

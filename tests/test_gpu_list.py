"""GPU parity of the list form (models of more than 12 species in sparse
states, plain runs) against the CPU oracle, bit for bit: 13 to 32 species;
meshes of less than a chunk of 32 tets, of exactly one and with a remainder;
few and many molecules in the tets that hold any (bit-plane groups, more
Philox blocks than are listed at a time); sources everywhere, in a region and
nowhere, masks and rates changed between runs; states that fill up until half
of the tets are listed and on past the density at which a run leaves the form;
both occupancy modes and leave laws; counts set species by species; a clone;
recordings; a batch in between."""
import numpy as np
import pytest

import oracle
from oracle import END, OCC
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


def _model(S, source=1e-5):
    names = [f"S{i}" for i in range(S)]
    diff = [1e-11 / (1 + 2 * i) for i in range(S)]
    diff[3] = diff[S - 1] = 0.0
    reac = [([], [names[0]], source), ([names[0]], [names[1]], 300.0), ([names[1], names[2]], [names[3]], 3e7),
            ([names[0], names[0]], [names[2]], 2e7), ([names[3]], [names[1], names[2]], 200.0),
            ([names[S - 1]], [names[12], names[0]], 100.0)]
    return I.model_from_lists(names, diff, reac if source else reac[1:])


def _sparse(rng, S, nt, share, values):
    c = np.zeros((S, nt), np.int32)
    n = max(1, int(share * nt))
    for _ in range(n):
        c[rng.integers(0, S), rng.integers(0, nt)] = rng.choice(values)
    return c


def _pair(capi, S, grid, share, values, occ=OCC, leave=0, source=1e-5, seed=5):
    verts, tets = I.kuhn_box_mesh(*grid, 0.5 * I.UM)
    nt = tets.shape[0]
    m = _model(S, source)
    counts = _sparse(np.random.default_rng(100 * S + nt), S, nt, share, values)
    g = capi.Simulation(verts, tets, m, seed, occupancy=occ, leave_law=leave, specialize=1)
    o = oracle.OracleSim(verts, tets, m, seed=seed, occ=occ, prec=32, leave=leave)
    for obj in (g, o):
        obj.set_counts(counts)
    assert g.specialized and g.tau == o.tau
    return g, o, counts


def _run(g, o, windows):
    t = o.time + windows * o.tau
    g.run(t)
    o.run(t)
    assert g.windows == o.windows and np.array_equal(g.get_counts(), o.get_counts())


@pytest.mark.parametrize("S", [13, 16, 20, 32])
@pytest.mark.parametrize("grid", [(5, 1, 1), (16, 1, 1), (9, 5, 4)])
def test_sizes(capi, S, grid):
    """30, 96 and 1,080 tets; a masked source."""
    g, o, _ = _pair(capi, S, grid, 0.1, [1, 2, 3])
    on = np.zeros(g.nt, np.uint8)
    on[: g.nt // 10 + 1] = 1
    for obj in (g, o):
        obj.set_reac_mask(0, on)
    _run(g, o, 20.4)
    _run(g, o, 3.0)


@pytest.mark.parametrize("occ", [OCC, END])
@pytest.mark.parametrize("leave", [0, 1])
def test_modes_and_heavy_tets(capi, occ, leave):
    """Few tets hold much: groups of 32 and word streams over several rounds of
    the block list, then the spread of the molecules over the mesh."""
    g, o, _ = _pair(capi, 20, (9, 6, 5), 0.15, [15, 16, 31, 33, 64, 400], occ=occ, leave=leave, source=0.0)
    for w in (1.0, 1.0, 2.5, 30.0):
        _run(g, o, w)
    g, o, _ = _pair(capi, 32, (9, 6, 5), 0.0, [1], occ=occ, leave=leave, source=0.0)
    c = np.zeros((32, g.nt), np.int32)
    c[:8, :32] = 15  # 30 Philox blocks in each of 32 tets that one chunk holds
    for obj in (g, o):
        obj.set_counts(c)
    _run(g, o, 4.3)


def test_filling_up_and_sources_everywhere(capi):
    """A source in every tet: from an empty mesh past half of the tets listed,
    past the density at which the next run leaves the form, with a rate change."""
    g, o, _ = _pair(capi, 14, (10, 5, 5), 0.0, [1], source=3e-6)
    for obj in (g, o):
        obj.set_counts(np.zeros((14, g.nt), np.int32))
    for k in (1e-6, 3e-6, 3e-5, 0.0):
        g.set_reac_rate(0, k)
        o.set_reac_rate(0, k)
        _run(g, o, 40.0)
    assert o.get_counts().sum() > g.nt


def test_masks_single_species_clone_batch_and_long_run(capi):
    g, o, counts = _pair(capi, 16, (8, 8, 6), 0.05, [1, 2])
    rng = np.random.default_rng(1)
    for _ in range(3):  # the sources move between runs
        on = (rng.random(g.nt) < 0.05).astype(np.uint8)
        for obj in (g, o):
            obj.set_reac_mask(0, on)
        _run(g, o, 7.7)
    b = capi.Batch([g], block=256)  # windows in another form in between
    t = o.time + 5 * o.tau
    b.run([t])
    o.run(t)
    _run(g, o, 3.0)
    b.close()
    c = g.clone(9)
    o2 = oracle.OracleSim(*I.kuhn_box_mesh(8, 8, 6, 0.5 * I.UM), _model(16), seed=9, occ=OCC, prec=32)
    o2.set_counts(counts)
    o2.set_reac_mask(0, on)
    for s in range(16):
        capi.steps_set_counts(c._sim, s, counts[s])
    _run(c, o2, 150.0)   # the list is built afresh on the way
    _run(c, o2, 1100.0)  # and looked at


def test_recordings(capi):
    import torch
    g, o, _ = _pair(capi, 20, (8, 6, 6), 0.08, [1, 2, 5], source=0.0)
    tets = np.arange(0, g.nt, 7, dtype=np.int32)
    buf = torch.zeros((10, 2, tets.size), dtype=torch.int32, device="cuda")
    dt = 3.3 * o.tau
    n = g.run_record(10.5 * dt, dt, np.array([0, 5], np.int32), tets, buf.data_ptr(), 10)
    assert n == 10
    rec = buf.cpu().numpy()
    for k in range(10):
        o.run((k + 1) * dt)
        assert np.array_equal(rec[k], o.get_counts()[[0, 5]][:, tets])


def test_batch_of_listed_and_other_members(capi):
    """A batch whose members are in sparse and in dense states (list form and warp
    tiles in one window), over two runs and then alone."""
    pairs = [_pair(capi, 14, (9, 6, 5), 0.1, [1, 2], seed=3), _pair(capi, 14, (6, 6, 5), 0.05, [1, 40], seed=4)]
    g, o, _ = _pair(capi, 14, (8, 5, 5), 0.1, [1], seed=6)
    c = np.random.default_rng(3).integers(0, 6, (14, g.nt)).astype(np.int32)
    for obj in (g, o):
        obj.set_counts(c)
    pairs.append((g, o, c))
    b = capi.Batch([p[0] for p in pairs], block=256, specialize=1)
    for k in (20.4, 21.7):
        ends = [p[1].time + k * p[1].tau for p in pairs]
        b.run(ends)
        for (g, o, _), t in zip(pairs, ends):
            o.run(t)
            assert g.windows == o.windows and np.array_equal(g.get_counts(), o.get_counts())
    b.close()
    for g, o, _ in pairs:
        _run(g, o, 5.5)

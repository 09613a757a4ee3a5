"""GPU parity of the warp-tile step (models of up to 12 species, on the
model-specialised kernels and on those for models given at run time) against the CPU oracle, bit for bit, where its
tiles, queues and packed tables have edges: meshes that end inside, at and
just past a warp's 32 tets and a block's 256; 1 to 13 species (the table of
words per species holds four to a word; 13 is the first model on the other
kernel); counts around the bit-plane threshold and its groups of 32, tets of
more than 127 words, chunks of more Philox blocks than are listed at a time;
reactions of every order, several events per tet, an immobile species, a
masked source; both occupancy modes, both leave laws, both launch forms."""
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


def _model(S):
    names = [f"S{i}" for i in range(S)]
    diff = [1e-11 / (1 + 3 * i) for i in range(S)]
    if S > 2:
        diff[2] = 0.0
    n = lambda i: names[i % S]  # noqa: E731
    reac = [([], [n(0)], 1e-4), ([n(0)], [n(1)], 300.0), ([n(1), n(2)], [n(3)], 3e6), ([n(0), n(0)], [n(2)], 2e6),
            ([n(3)], [n(1), n(2)], 200.0), ([n(S - 1)], [], 50.0)]
    return I.model_from_lists(names, diff, reac)


def _check(capi, S, grid, values, occ=OCC, leave=0, flow=False, block=256, mask=True, windows=(3.0, 5.4)):
    _check_kernel(capi, S, grid, values, occ, leave, flow, block, mask, windows, 1)
    if leave == 0 and not (flow and block != 256):  # the kernels for models given at run time
        _check_kernel(capi, S, grid, values, occ, leave, flow, block, mask, windows, -1)


def _check_kernel(capi, S, grid, values, occ, leave, flow, block, mask, windows, specialize):
    verts, tets = I.kuhn_box_mesh(*grid, 0.5 * I.UM)
    nt = tets.shape[0]
    m = _model(S)
    rng = np.random.default_rng(S * 1000 + nt)
    counts = rng.choice(np.asarray(values, np.int32), size=(S, nt)).astype(np.int32)
    on = (rng.random(nt) < 0.5).astype(np.uint8)
    g = capi.Simulation(verts, tets, m, 7, occupancy=occ, leave_law=leave, specialize=specialize, flow=flow,
                        block=block)
    o = oracle.OracleSim(verts, tets, m, seed=7, occ=occ, prec=32, leave=leave)
    for obj in (g, o):
        obj.set_counts(counts)
        if mask:
            obj.set_reac_mask(0, on)
    assert g.specialized == (specialize > 0) and g.tau == o.tau
    for k in windows:
        g.run(k * o.tau)
        o.run(k * o.tau)
        assert np.array_equal(g.get_counts(), o.get_counts())
    assert o.events > 0


SPARSE = [0, 0, 0, 1, 2, 5]
EDGES = [0, 1, 14, 15, 16, 17, 31, 32, 33, 63, 64, 65, 400]


@pytest.mark.parametrize("S", [1, 2, 4, 5, 8, 9, 12, 13])
def test_species_counts(capi, S):
    _check(capi, S, (6, 3, 2), SPARSE)
    _check(capi, S, (6, 3, 2), EDGES, mask=False)


@pytest.mark.parametrize("grid", [(1, 1, 1), (5, 1, 1), (16, 1, 1), (11, 4, 1), (43, 1, 1), (8, 8, 8)])
@pytest.mark.parametrize("flow", [False, True])
def test_mesh_sizes(capi, grid, flow):
    """6, 30, 96 (three full warps), 264, 258 and 3,072 (twelve full blocks) tets."""
    _check(capi, 5, grid, SPARSE + EDGES, flow=flow)


@pytest.mark.parametrize("occ", [OCC, END])
@pytest.mark.parametrize("leave", [0, 1])
@pytest.mark.parametrize("block", [64, 512])
def test_modes(capi, occ, leave, block):
    _check(capi, 10, (7, 3, 5), SPARSE + EDGES, occ=occ, leave=leave, block=block, flow=leave == 0)


@pytest.mark.parametrize("leave", [0, 1])
def test_long_word_streams(capi, leave):
    """Twelve species of up to 15 molecules: up to 180 words in a tet, more
    Philox blocks in 32 tets than are listed at a time."""
    _check(capi, 12, (5, 5, 3), [13, 14, 15], leave=leave, windows=(1.0, 2.3))
    _check(capi, 12, (5, 5, 3), [9, 10, 11], leave=leave, windows=(1.0, 2.3))


@pytest.mark.parametrize("cells,lanes", [(809, 4), (810, 8), (1618, 8), (1619, 16), (3237, 16), (3238, 32)])
@pytest.mark.parametrize("S", [3, 6])
def test_tets_per_warp(capi, cells, lanes, S):
    """Models given at run time on either side of the sizes (4,856, 9,712 and
    19,424 tets) below which a warp takes fewer tets, all with a ragged end."""
    assert (6 * cells + lanes - 1) // lanes >= 608 or lanes == 4
    _check_kernel(capi, S, (cells, 1, 1), SPARSE + EDGES, OCC, 0, False, 256, True, (2.0, 3.3), -1)

"""Rates beyond the float range (the library takes any finite double; the kernels
use float rates): a reaction whose reactant is absent never fires, and the
others fire as if it were not there. Bit for bit against the model without it,
on the oracle, in the kernels for models given at run time and in compiled ones."""
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


@pytest.mark.parametrize("specialize", [-1, 1])
@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("lhs", [["X"], ["X", "A"], ["X", "X"]])
@pytest.mark.parametrize("place", [0, 1, 2])
def test_absent_reactant_of_an_infinite_rate(capi, specialize, flow, lhs, place):
    """One A (immobile) in half of the tets, so that a tet fires at most once per
    window; the reaction that cannot fire stands before, between and after
    the two that can."""
    names = ["A", "B", "C", "X", "W"]
    diff = [0.0, 0.0, 0.0, 1e-11, 1e-11]
    reac = [(["A"], ["B"], 400.0), (["A"], ["C"], 200.0)]
    never = (lhs, ["B"], 1e39 if len(lhs) == 1 else 1e300)
    model = I.model_from_lists(names, diff, reac[:place] + [never] + reac[place:])
    verts, tets = I.kuhn_box_mesh(6, 5, 3, 0.5 * I.UM)
    counts = np.zeros((5, tets.shape[0]), np.int32)
    counts[0, ::2] = 1
    counts[4] = 3
    o = oracle.OracleSim(verts, tets, I.model_from_lists(names, diff, reac), seed=8, occ=oracle.OCC, prec=32)
    g = capi.Simulation(verts, tets, model, 8, specialize=specialize, flow=flow)
    for obj in (g, o):
        obj.set_counts(counts)
    for k in (6.0, 15.4):
        g.run(k * o.tau)
        o.run(k * o.tau)
        assert np.array_equal(g.get_counts(), o.get_counts())
    assert o.events > 20


@pytest.mark.parametrize("form", ["list", "tiles", "flow", "run-time", "run-time flow", "batch"])
@pytest.mark.parametrize("S", [6, 14])
@pytest.mark.parametrize("lhs", [["X", "Y"], ["X", "X"]])
def test_reactants_of_an_infinite_rate_that_never_meet(capi, form, S, lhs):
    """One X or one Y stands in different tets of every warp and chunk, each beside
    an A: a reaction of both, or of two X, can fire nowhere, and A's fire as in
    the model without it, in every form of the step."""
    names = ["A", "B", "C", "X", "Y"] + [f"W{i}" for i in range(S - 5)]
    diff = [0.0] * 5 + [1e-11] * (S - 5)
    reac = [(["A"], ["B"], 400.0), (["A"], ["C"], 200.0)]
    model = I.model_from_lists(names, diff, reac[:1] + [(lhs, ["B"], 1e300)] + reac[1:])
    verts, tets = I.kuhn_box_mesh(9, 5, 4, 0.5 * I.UM)
    nt = tets.shape[0]
    counts = np.zeros((S, nt), np.int32)
    counts[0, ::10] = 1
    counts[3, ::20] = 1
    counts[4, 10::20] = 1
    if form != "list":
        counts[5] = 3
    o = oracle.OracleSim(verts, tets, I.model_from_lists(names, diff, reac), seed=8, occ=oracle.OCC, prec=32)
    g = capi.Simulation(verts, tets, model, 8, specialize=-1 if form.startswith("run-time") else 1,
                        flow="flow" in form, reorder=capi.STEPS_REORDER_NONE)
    for obj in (g, o):
        obj.set_counts(counts)
    b = capi.Batch([g], block=256, specialize=1) if form == "batch" else None
    for k in (6.0, 15.4):
        if b:
            b.run([k * o.tau])
        else:
            g.run(k * o.tau)
        o.run(k * o.tau)
        assert np.array_equal(g.get_counts(), o.get_counts())
    assert o.events > 20

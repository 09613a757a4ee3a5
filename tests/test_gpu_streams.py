"""Simulations and batches on a stream of their own while the default stream is
busy: everything a run reads is written in the order of its own stream, so the
counts equal the oracle's whatever the default stream still has to do, and
nothing it does later changes them."""
import numpy as np
import pytest

import oracle
from paper_1610_02258_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BUSY = 40_000_000  # clock cycles the default stream sleeps, about 20 ms


@pytest.fixture(scope="module")
def capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_02258_gb300.build import build
    build()
    from paper_1610_02258_gb300 import capi as c
    return c


def _busy():
    import torch
    torch.cuda.current_stream().synchronize()
    torch.cuda._sleep(BUSY)


def _oracle(w, t_ends, seed, leave=0, masks=None):
    o = oracle.OracleSim(w.verts, w.tets, w.model, seed=seed, occ=oracle.OCC, prec=32, leave=leave)
    o.set_counts(w.counts)
    for r, m in (masks or {}).items():
        o.set_reac_mask(r, m)
    for t in t_ends:
        o.run(t)
    return o.get_counts()


@pytest.mark.parametrize("specialize", [1, -1])
def test_first_flow_run(capi, specialize):
    """The finished-window words of a first flow launch are zero before it
    starts, though the memory held those of a simulation that ran longer."""
    import torch
    w = I.config2(nx=4, t_end=1.5e-3)
    side = torch.cuda.Stream()
    for seed in (3, 4, 5):
        g = capi.Simulation(w.verts, w.tets, w.model, seed, specialize=specialize, flow=True,
                            cuda_stream=side.cuda_stream)
        g.set_counts(w.counts)
        t = (5 - seed + 1) * 0.5e-3  # each shorter than the one before it
        _busy()
        g.run(t)
        first = g.get_counts()
        torch.cuda.synchronize()
        assert np.array_equal(first, _oracle(w, [t], seed))
        g.close()


def test_first_batch_flow_run(capi):
    import torch
    ws = [I.config2(seed=40 + j, nx=4, t_end=1e-3) for j in range(3)]
    side = torch.cuda.Stream()
    for t in (1e-3, 0.5e-3):
        members = [capi.from_workload(w) for w in ws]
        b = capi.Batch(members, block=256, specialize=1, flow=True, cuda_stream=side.cuda_stream)
        _busy()
        b.run([t] * len(ws))
        for w, m in zip(ws, members):
            assert np.array_equal(m.get_counts(), _oracle(w, [t], w.seed))
        b.close()


@pytest.mark.parametrize("leave", [0, 1])
def test_setup_while_the_default_stream_is_busy(capi, leave):
    """A simulation created, masked, filled, run and cloned on a side stream. The
    tets keep their order, so that no upload follows the zeroed counts."""
    import torch
    w = I.config2(nx=2, t_end=1.5e-3)
    on = (np.arange(w.tets.shape[0]) % 3 != 0).astype(np.uint8)
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    ends = [0.7e-3, 1.5e-3]
    want = _oracle(w, ends, 9, leave, {0: on})
    _busy()
    g = capi.Simulation(w.verts, w.tets, w.model, 9, reorder=capi.STEPS_REORDER_NONE, leave_law=leave,
                        cuda_stream=side.cuda_stream)
    _busy()
    g.set_reac_mask(0, on)
    g.set_counts(w.counts)
    c = g.clone(9, cuda_stream=other.cuda_stream)
    c.set_counts(w.counts)
    for t in ends:
        g.run(t)
        c.run(t)
    torch.cuda.synchronize()
    assert np.array_equal(g.get_counts(), want)
    assert np.array_equal(c.get_counts(), want)


def test_batch_while_the_default_stream_is_busy(capi):
    import torch
    ws = [I.config1(seed=50 + j) for j in range(3)]
    side = torch.cuda.Stream()
    members = [capi.from_workload(w, cuda_stream=side.cuda_stream) for w in ws]
    _busy()
    b = capi.Batch(members, block=64, cuda_stream=side.cuda_stream)
    b.run([w.t_end for w in ws])
    torch.cuda.synchronize()
    for w, m in zip(ws, members):
        assert np.array_equal(m.get_counts(), _oracle(w, [w.t_end], w.seed))

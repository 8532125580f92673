"""A step begun by its phases and left before its decode must leave nothing
behind: whatever replaces the state or starts the next step, the result is
that of a handle that never saw the abandoned step, bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

L = 7


def _begin(sim):
    """Every phase up to the update."""
    sim.encode()
    sim.flag()
    sim.traverse()
    sim.fv1()


def _equal(a, b, leaves=True):
    ga, gb = a.fields(), b.fields()
    for q in ("h", "qx", "qy"):
        assert np.array_equal(ga[q], gb[q]), q
    if leaves:
        assert np.array_equal(a.leaves(), b.leaves())
    assert a.time()[:2] == b.time()[:2]


@pytest.mark.parametrize("matched", [False, True])
@pytest.mark.parametrize("how", ["set_fields", "load", "uniform"])
@pytest.mark.parametrize("precision", [64, 32])
def test_a_new_state_after_an_abandoned_step(matched, how, precision):
    from paper_2206_05761_gb300.sim import Simulation
    p, f = synth.bumpy_dam_break(L=L, eps=1e-3, seed=5)
    g = synth.bumpy_dam_break(L=L, eps=1e-3, seed=9)[1]
    # the first state is rough, every finest cell a leaf; the second is coarse in part
    p = dict(p, flux_match=matched)
    rough = dict(f)
    rng = np.random.default_rng(1)
    rough["h"] = rng.uniform(0.5, 1.0, f["h"].shape)
    if precision == 32:
        g = {k: v.astype(np.float32).astype(np.float64) for k, v in g.items()}
    other = dict(h=g["h"], qx=g["qx"], qy=g["qy"], z=f["z"])
    a = Simulation(p, dict(rough, z=f["z"]), precision)
    b = Simulation(p, other, precision)
    _begin(a)
    if how == "load":
        a.load(b.save())
    else:
        a.set_fields(other)
    a.set_time(0.0, 1e-3)
    b.set_time(0.0, 1e-3)
    for s in (a, b):
        if how == "uniform":
            s.advance_uniform(max_steps=2)
        else:
            s.advance(max_steps=2)
    if how != "uniform":
        assert 4 ** L > len(b.leaves()) > 0
    _equal(a, b, leaves=how != "uniform")
    a.close()
    b.close()


@pytest.mark.parametrize("matched", [False, True])
@pytest.mark.parametrize("what", ["step twice", "phases again", "advance", "profile_step", "profile_update"])
@pytest.mark.parametrize("precision", [64, 32])
def test_a_step_begun_again(matched, what, precision):
    # every finest cell is a wet leaf, so that two queues do not fit one list
    import paper_2206_05761_gb300.hwfv1 as H
    from paper_2206_05761_gb300.sim import Simulation
    p, f = synth.bumpy_dam_break(L=L, eps=0.0, seed=5)
    p = dict(p, flux_match=matched)
    f = dict(f, h=np.random.default_rng(1).uniform(0.5, 1.0, f["h"].shape))
    a, b = Simulation(p, f, precision), Simulation(p, f, precision)
    _begin(a)
    if what == "step twice":
        a.fv1()
        a.decode()
    elif what == "phases again":
        a.step()
    elif what == "advance":
        a.advance(max_steps=1)
    elif what == "profile_step":
        H.hwfv1_profile_step(a.hd)
    else:
        H.hwfv1_profile_update(a.hd, 3)
    b.step()
    _equal(a, b)
    ca, cb = a.counters(), b.counters()
    assert ca[0] == cb[0] == 1 and ca[1] == cb[1] == 4 ** L
    assert ca[3] == cb[3] == 4 ** L                # full updates: the list's length
    a.close()
    b.close()


@pytest.mark.parametrize("precision", [64, 32])
def test_the_update_after_uniform_steps_has_no_leaves(precision):
    # before any traversal: nothing is listed, so nothing is updated or queued
    from paper_2206_05761_gb300.sim import Simulation
    p, f = synth.bumpy_dam_break(L=L, eps=1e-3, seed=5)
    a, b = Simulation(p, f, precision), Simulation(p, f, precision)
    for s in (a, b):
        s.advance_uniform(max_steps=2)
    a.fv1()
    _equal(a, b, leaves=False)
    for s in (a, b):
        s.advance(max_steps=2)
    _equal(a, b)
    assert a.counters()[:4] == b.counters()[:4]
    a.close()
    b.close()

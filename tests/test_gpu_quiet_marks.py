"""The marks of tiles that hold only +0 across everything that moves the state
between two new states: uniform steps, a load, the skip modes, the phase
calls.  The run with marks equals the full sweep bit for bit throughout."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

L = 8


def _column(p, cx, cy, speed):
    x, y = synth.centres(p)
    h = np.where((x - cx) ** 2 + (y - cy) ** 2 < 0.01, 0.7, 0.0)
    return dict(h=h, qx=h * speed, qy=np.zeros_like(h))


@pytest.mark.parametrize("between", ["uniform", "load", "store", "levels", "phases", "abandoned"])
def test_marks_hold_across(between):
    from paper_2206_05761_gb300.sim import Simulation
    p, f = synth.dry_bed_dam_break(L=L, eps=1e-3)
    a, b = Simulation(p, f), Simulation(dict(p, full_sweep=True), f)
    first = a.save()
    states = [_column(p, 0.8, 0.7, 0.0), _column(p, 0.5, 0.1, 1.0), {k: f[k] for k in ("h", "qx", "qy")}]
    for k, s in enumerate(states):
        for sim in (a, b):
            sim.advance(max_steps=3)
            if between == "uniform":
                sim.advance_uniform(max_steps=2)
            elif between == "load":
                sim.load(first)
            elif between == "store":
                sim.set_leaf_store(True)
                sim.advance(max_steps=3)
                sim.set_leaf_store(False)
            elif between == "levels":
                # the finest level everywhere: the skip's own encode, the plain step's result
                sim.set_skip_levels(np.full((1 << (L - 4),) * 2, L), audit_K=2)
                sim.advance(max_steps=3)
                sim.set_skip_levels(None)
            elif between == "phases":
                sim.step()
                sim.step()
            else:
                sim.encode()
                sim.flag()
                sim.traverse()
                sim.fv1()
            sim.set_fields(s)
            sim.set_time(0.0, 1e-3)
        g = a.fields()
        for q in ("h", "qx", "qy"):
            assert np.array_equal(g[q], s[q]), (k, q)
        for n in (1, 5):
            a.advance(max_steps=n)
            b.advance(max_steps=n)
            ga, gb = a.fields(), b.fields()
            for q in ("h", "qx", "qy"):
                assert np.array_equal(ga[q], gb[q]), (k, n, q)
            assert np.array_equal(a.leaves(), b.leaves())
            assert a.time() == b.time()
    a.close()
    b.close()

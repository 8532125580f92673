"""hwfv1_set_fields and hwfv1_get_fields: the layout conversion at the edges
of its tiles (one parent, part of a tile, one tile, many) and for pointers of
8-byte alignment, and the quiescence marks that survive a new state: a run
that goes on from it must equal the full sweep bit for bit."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 3, 5, 6, 8])
@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("offset", [0, 1])
def test_fields_in_and_out(L, precision, offset):
    import paper_2206_05761_gb300.hwfv1 as H
    from paper_2206_05761_gb300.sim import Simulation
    p, f = synth.circular_dam_break(L=L, eps=1e-3)
    sim = Simulation(p, f, precision)
    n = 1 << (2 * L)
    new = [synth.random_state(L, 40 + q).reshape(-1) for q in range(3)]
    new[0] = np.abs(new[0])
    if precision == 32:
        new = [a.astype(np.float32).astype(np.float64) for a in new]
    src = []
    for a in new:
        t = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
        t[offset:offset + n] = torch.from_numpy(a)
        src.append(t)
    torch.cuda.synchronize()
    H.hwfv1_set_fields(sim.hd, *[t[offset:offset + n] for t in src])
    _, smax = sim.stats()
    assert smax == [max(1.0, float(np.abs(a).max())) for a in new]
    out = [torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    H.hwfv1_get_fields(sim.hd, out[0][offset:offset + n], None, out[2][offset:offset + n])
    torch.cuda.synchronize()
    for q in (0, 2):
        got = out[q].cpu().numpy()
        assert np.array_equal(got[offset:offset + n], new[q])
        assert np.all(got[:offset] == 7.0) and np.all(got[offset + n:] == 7.0)
    assert torch.all(out[1] == 7.0)
    sim.close()


@pytest.mark.parametrize("relief", [0.0, 0.05])
@pytest.mark.parametrize("L", [7, 11])
def test_a_new_state_keeps_only_true_quiescence_marks(L, relief):
    from paper_2206_05761_gb300.sim import Simulation
    p, f = synth.dry_bed_dam_break(L=L, eps=1e-3, relief=relief)
    p2 = dict(p, full_sweep=True)
    a, b = Simulation(p, f), Simulation(p2, f)
    x, y = synth.centres(p)
    states = [f]
    for cx, cy, speed in ((0.8, 0.7, 0.0), (0.5, 0.1, 1.0)):       # water moves to ground that was dry, and back
        h = np.where((x - cx) ** 2 + (y - cy) ** 2 < 0.01, 0.7, 0.0)
        states.append(dict(h=h, qx=h * speed, qy=np.zeros_like(h)))
    states.append(f)
    for k, s in enumerate(states):
        if k:
            a.set_fields(s)
            b.set_fields(s)
            g = a.fields()
            for q in ("h", "qx", "qy"):
                assert np.array_equal(g[q], s[q]), (k, q)
        for n in (1, 7 if L == 11 else 24):
            a.advance(max_steps=n)
            b.advance(max_steps=n)
            ga, gb = a.fields(), b.fields()
            for q in ("h", "qx", "qy"):
                assert np.array_equal(ga[q], gb[q]), (k, n, q)
            assert np.array_equal(a.leaves(), b.leaves())
            assert a.time() == b.time()
    a.close()
    b.close()

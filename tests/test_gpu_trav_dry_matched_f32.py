"""The fused traversal and dry pass with matched fluxes in float32 against the
kernels of the phases, which a profiled step runs: the same bits."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


# a CTA per quarter tile, per tile, and the work list; with dry ground and inflow
@pytest.mark.parametrize("scene,L", [("bumps", 1), ("bumps", 5), ("bumps", 8), ("bumps", 11), ("dry bed", 7),
                                     ("inflow", 6)])
def test_matched_float32(scene, L):
    import paper_2206_05761_gb300.hwfv1 as H
    from paper_2206_05761_gb300.sim import Simulation
    if scene == "bumps":
        p, f = synth.bumpy_dam_break(L=L, eps=1e-3, seed=5)
    elif scene == "dry bed":
        p, f = synth.dry_bed_dam_break(L=L, eps=1e-3, relief=0.05)
    else:
        p, f = synth.inflow_basin(L=L, eps=1e-3, q=0.01)
    p = dict(p, flux_match=True)
    a, b = Simulation(p, f, 32), Simulation(p, f, 32)
    d = Simulation(p, f, 64)
    for n in (1, 4):
        a.advance(max_steps=n)
        for _ in range(n):
            H.hwfv1_profile_step(b.hd)
        ga, gb = a.fields(), b.fields()
        for q in ("h", "qx", "qy"):
            assert np.array_equal(ga[q], gb[q]), (n, q)
        assert np.array_equal(a.leaves(), b.leaves())
        assert a.time() == b.time()
        assert a.counters()[:4] == b.counters()[:4]
        if n == 1:
            # one step from the same state in float64: a few float roundings of
            # sums of some twenty terms no larger than the fields' scale
            d.advance(max_steps=1)
            gd = d.fields()
            if np.array_equal(a.leaves(), d.leaves()):
                for q in ("h", "qx", "qy"):
                    scale = max(1.0, np.abs(gd["h"]).max(), np.abs(gd[q]).max())
                    assert np.abs(ga[q] - gd[q]).max() <= 64 * 2.0 ** -24 * 10 * scale, q
    for s in (a, b, d):
        s.close()

"""The step's fused traversal and dry pass (a CTA per tile up to eight tiles an
SM, a work list beyond) against the kernels of the phases, which a profiled
step runs: the same fields, leaves, time and counters, bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _case(scene, L):
    if scene == "dry bed":
        return synth.dry_bed_dam_break(L=L, eps=1e-3, relief=0.05)
    if scene == "inflow":
        return synth.inflow_basin(L=L, eps=1e-3, q=0.01)
    p, f = synth.bumpy_dam_break(L=L, eps=1e-2 if scene == "coarse" else 0.0, seed=5)
    return (dict(p, flux_match=True) if scene == "matched" else p), f


@pytest.mark.parametrize("scene,L", [("dry bed", 1), ("dry bed", 2), ("dry bed", 6), ("dry bed", 9), ("dry bed", 11),
                                     ("inflow", 5), ("inflow", 7), ("coarse", 4), ("coarse", 10), ("coarse", 11),
                                     ("all leaves", 5), ("all leaves", 8), ("matched", 7)])
@pytest.mark.parametrize("precision", [64, 32])
def test_fused_step_equals_the_phases(scene, L, precision):
    import paper_2206_05761_gb300.hwfv1 as H
    from paper_2206_05761_gb300.sim import Simulation
    if scene == "matched" and precision == 32:
        pytest.skip("matched fluxes are float64")
    p, f = _case(scene, L)
    a, b = Simulation(p, f, precision), Simulation(p, f, precision)
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
    a.close()
    b.close()

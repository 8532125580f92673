"""Manning friction on cells whose values leave the range of the integer
float64 arithmetic, element by element: the update of the first step from one
state on both sides.

The depths hold no friction term and are the oracle's bits.  A discharge is
q (1/D) with D = 1 + x and x within 2^-40 relative (the Newton step of the
inverse cube root; the quotient as written, within a few units in the last
place, outside the float range), so within 2^-40 + 8 * 2^-53 relative, plus
four units of the smallest subnormal where the product is subnormal."""
import numpy as np
import pytest

import oracle

from test_gpu_extreme_values import CASES, extreme_case
from test_gpu_parity import _sim

pytestmark = pytest.mark.gpu

RTOL = 2.0 ** -40 + 8 * 2.0 ** -53
ATOL = 4 * 2.0 ** -1074


def _one_step(p, f):
    sim, ref = _sim(p, f), oracle.State(p, f)
    sim.advance(max_steps=1)
    ref.step()
    g = sim.fields()
    dt = sim.time()[1]
    sim.close()
    return g, dt, ref


@pytest.mark.parametrize("name", [None] + sorted(CASES))
@pytest.mark.parametrize("L", [3, 6])
@pytest.mark.parametrize("n_M", [0.03, 1e3])
def test_friction_element_by_element(name, L, n_M):
    if name is None:
        p, f = extreme_case(L, 0, 0, 1e-6)
    else:
        p, f = extreme_case(L, **CASES[name])
    free = _one_step(p, f)[0]
    p = dict(p, manning_n=n_M)
    g, dt, ref = _one_step(p, f)
    assert np.array_equal(g["h"], ref.h)
    for k in ("qx", "qy"):
        o = getattr(ref, k)
        assert np.isfinite(o).all()
        off = np.abs(g[k] - o) - ATOL
        assert np.all(off <= RTOL * np.abs(o)), (k, np.nanmax(off / np.maximum(np.abs(o), ATOL)))
    if name is None:
        # the friction term takes part: discharges move by its share
        assert np.mean(g["qx"] != free["qx"]) > 0.5
    # the bound's speeds are |q (1/h)| + sqrt(g h): as far off as the discharges
    assert abs(dt - ref.dt) <= 2 * RTOL * ref.dt

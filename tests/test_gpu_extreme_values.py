"""Cells whose values leave the range of the integer float64 arithmetic (depths
and discharges whose products are subnormal, underflow, or lie near the top of
the exponent range), next to ordinary cells in the same warps: the flux and the
update must give the oracle's bits on either path, and with friction the
oracle's values."""
import numpy as np
import pytest

import synth

from test_gpu_parity import one_step_parity

pytestmark = pytest.mark.gpu


def extreme_case(L, h2, q2, tol, n_M=0.0, spread=False):
    """Random wet cells; depths times 2^h2 and discharges times 2^q2, in all
    cells, or (spread) in cells picked at random with exponents up to these."""
    p, _ = synth.bumpy_dam_break(L=L, eps=0.0, seed=3)
    p = dict(p, tol_h=tol, n_M=n_M)
    n = 1 << L
    rng = np.random.default_rng(L + 7)
    h = rng.uniform(0.5, 1.0, (n, n))
    qx, qy = (rng.uniform(-1.0, 1.0, (n, n)) for _ in range(2))
    eh, eq = np.full((n, n), h2), np.full((n, n), q2)
    if spread:
        pick = rng.random((n, n)) < 0.1
        w = rng.random((n, n))
        eh, eq = np.where(pick, (h2 * w).astype(int), 0), np.where(pick, (q2 * w).astype(int), 0)
    zero = rng.random((n, n)) < 0.05
    qx[zero] = 0.0
    qy[zero] = -0.0
    return p, dict(h=np.ldexp(h, eh), qx=np.ldexp(qx, eq), qy=np.ldexp(qy, eq), z=np.zeros((n, n)))


CASES = {
    "subnormal discharges": dict(h2=0, q2=-1070, tol=1e-6, spread=True),
    "squares underflow": dict(h2=0, q2=-530, tol=1e-6, spread=True),
    "tiny depths": dict(h2=-530, q2=-795, tol=2.0 ** -600),
    "tiny and ordinary depths": dict(h2=-500, q2=-900, tol=2.0 ** -510, spread=True),
    "huge depths": dict(h2=404, q2=606, tol=1e-6),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("L", [3, 6])
@pytest.mark.parametrize("pre_steps", [0, 1])
def test_out_of_range_cells_match_the_oracle(name, L, pre_steps):
    p, f = extreme_case(L, **CASES[name])
    one_step_parity(p, f, pre_steps=pre_steps)


@pytest.mark.parametrize("name", ["subnormal discharges", "tiny depths"])
def test_out_of_range_cells_with_friction(name):
    p, f = extreme_case(5, **CASES[name], n_M=0.03)
    one_step_parity(p, f, exact=False)

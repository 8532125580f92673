"""Matched faces whose halves and quarters are refined to different depths on
all four sides (a few isolated spikes in still water: the tree refines to the
finest level next to leaves of any size), against the oracle, bit for bit."""
import numpy as np
import pytest

import synth

from test_gpu_parity import one_step_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [2, 3, 4, 6, 8])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_jumps_of_any_depth(L, seed):
    p, f = synth.circular_dam_break(L=L, eps=1e-2)
    rng = np.random.default_rng(seed)
    n = 1 << L
    h = np.full((n, n), 1.0)
    k = 1 if L <= 3 else 6
    h[rng.integers(0, n, k), rng.integers(0, n, k)] += rng.uniform(0.5, 2.0, k)
    q = [np.where(h > 1.0, rng.uniform(-1.0, 1.0, (n, n)), 0.0) for _ in range(2)]
    f = dict(f, z=np.zeros((n, n)), h=h, qx=q[0], qy=q[1])
    one_step_parity(dict(p, bc=("closed",) * 4, flux_match=True), f)

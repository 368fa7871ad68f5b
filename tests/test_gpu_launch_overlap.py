"""Launch-bound steps: a kernel's launch overlaps its predecessor without waiting grids piling up on the SMs."""
import time

import numpy as np
import pytest

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


def _step_seconds(ne, steps=7, reps=25):
    """Fastest of reps calls of `steps` fixed steps (2D, N = 1, FP64, default schedule)."""
    s = nsk.Solver(2, ne, 1)
    s.set_params()
    g = np.random.Generator(np.random.PCG64(0))
    E, npe = ne[0] * ne[1], 4
    rho = 1.0 + 1e-3 * g.standard_normal((E, npe))
    s.set_state(np.stack([rho, 0.0 * rho, 0.0 * rho, rho]))
    dt = s.compute_dt(0.01)
    best = np.inf
    for _ in range(reps):
        t0 = time.perf_counter()
        s.step(dt, steps)
        best = min(best, time.perf_counter() - t0)
    s.close()
    return best


def test_steps_of_a_few_hundred_blocks_stay_launch_bound():
    """Meshes of 400 to 6000 elements of N = 1 are launch-bound: 105 launches a call, a few us each, so the
    largest takes little longer than the smallest. Waiting grids that pile up on the SMs make the middle
    ones more than twice as slow as the smallest; the bound lies between."""
    small = _step_seconds((20, 20))
    for ne in ((80, 80), (109, 55)):
        assert _step_seconds(ne) < 1.6 * small, ne

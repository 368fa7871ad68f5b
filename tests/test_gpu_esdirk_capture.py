"""The implicit step where its Arnoldi steps cannot be captured into a graph: launched directly, the same results."""
import numpy as np
import pytest

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


CASES = [((64,), True), ((64,), False), ((1100,), False)]


def _both(ne, precond):
    """(state, statistics) of a step with and without graphs."""
    got = []
    for refuse in (False, True):
        s = nsk.Solver(1, ne, 3)
        s.set_params(kappa=1e-3, alpha=100.0, beta=1e-2, mu=1e-2)
        x = s.node_coords()[0]
        rho = 1.0 + 0.2 * np.sin(2 * np.pi * x)
        s.set_state(np.stack([rho, 0.01 * rho, rho]))
        dt = 20.0 * s.compute_dt(0.5)
        nsk._test_hook_esdirk_refuse_capture(refuse)
        try:
            stats = s.step_esdirk(dt, 1, newton_tol=1e-10, krylov_tol=1e-4, block_precond=precond)
        finally:
            nsk._test_hook_esdirk_refuse_capture(False)
        got.append((s.get_state(), stats))
        s.close()
    return got


@pytest.mark.parametrize("ne,precond", CASES)
def test_refused_capture_falls_back_to_launches(gpu, ne, precond):
    """The small systems' graph of four steps (up to 4096 values) and the large systems' graph of each step."""
    (a, sa), (b, sb) = _both(ne, precond)
    assert np.array_equal(a, b)
    assert all(sa[k] == sb[k] for k in ("newton", "krylov", "failed")) and sa["krylov"] > 4


@pytest.mark.parametrize("ne,precond", CASES)
def test_direct_launches_count_their_residuals_once(gpu, ne, precond):
    (_, sa), (_, sb) = _both(ne, precond)
    assert sa["rhs"] == sb["rhs"]

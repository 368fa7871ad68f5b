"""A tuned small context: every kind of call takes a schedule that suits it, also where the single-block
schedule, which runs the steps of a call in one launch, is the fastest for fixed steps."""
import time

import numpy as np
import pytest

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


def _solver(dim, ne, N):
    s = nsk.Solver(dim, ne, N)
    s.set_params(kappa=1e-3, alpha=100.0, beta=1e-2, mu=1e-2)
    g = np.random.Generator(np.random.PCG64(1))
    rho = 1.0 + 1e-3 * g.standard_normal(s.shape[1:])
    U = np.stack([rho] + [0.0 * rho] * dim + [rho])
    s.set_state(U)
    return s, U


def _fastest(f, reps=60):
    best = np.inf
    for _ in range(reps):
        t0 = time.perf_counter()
        f()
        best = min(best, time.perf_counter() - t0)
    return best


CASES = [(1, (64,), 3), (1, (128,), 3), (1, (100,), 2), (2, (4, 4), 3)]


@pytest.mark.parametrize("dim,ne,N", CASES)
@pytest.mark.parametrize("call", ["rhs", "adaptive", "fixed"])
def test_tuned_calls_take_the_fastest_schedule(gpu, dim, ne, N, call):
    """Tuned time against the best of all schedules set by hand, 15 % for the tuner's own noise."""
    import torch

    s, U = _solver(dim, ne, N)
    Ud, out = torch.from_numpy(U).to(gpu), torch.empty(s.shape, dtype=torch.float64, device=gpu)
    dt = s.compute_dt(0.1)

    def run():
        if call == "rhs":
            s.rhs(0.0, out)
        else:
            s.step(-0.1 if call == "adaptive" else dt, 4)

    hand = np.inf
    for tpb in (128, 256):
        for f in (0, 1, 2, 3):
            s.set_schedule(tpb, f)
            s.set_state(Ud)
            run()
            hand = min(hand, _fastest(run))
    tuned = []
    for _ in range(3):  # the best of three tunings: another program's moment on the host is not the tuner's choice
        s.set_state(Ud)
        s.autotune()
        run()
        tuned.append((_fastest(run), s.get_schedule()))
    assert min(tuned)[0] <= 1.15 * hand, (tuned, hand)
    s.close()


@pytest.mark.parametrize("dim,ne,N", CASES)
def test_results_do_not_depend_on_the_tuning(gpu, dim, ne, N):
    s, U = _solver(dim, ne, N)
    got = []
    for tuned in (False, True):
        s.set_state(U)
        if tuned:
            s.autotune()
        r = [s.rhs(), s.lift()]
        s.step(-0.1, 2)
        s.step(1e-5, 2)
        s.step_esdirk(1e-4, 1)
        got.append(r + [s.get_state()])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    s.close()


def test_schedules_set_by_hand_stay(gpu):
    """After set_schedule nothing of an earlier tuning is left: schedule 3 runs a residual in its one launch."""
    s, U = _solver(1, (64,), 3)
    s.autotune()
    s.set_schedule(256, 3)
    s.set_profiling(True)
    s.rhs()
    assert s.get_profile()["k_block"][1] == 1
    assert s.get_schedule() == (256, 3)
    s.close()


@pytest.mark.parametrize("dim,ne,N", [(2, (24, 24), 3), (3, (6, 6, 6), 4)])
def test_tuner_reports_the_blocks_that_run(gpu, dim, ne, N):
    """FP64, N >= 3, 2D and 3D: schedules 0 and 1 run 128-thread blocks, so that is what the tuner reports."""
    s, _ = _solver(dim, ne, N)
    for _ in range(12):
        s.set_schedule(256, 0)
        tpb, fused, _ = s.autotune()
        assert fused not in (0, 1) or tpb == 128
    s.close()

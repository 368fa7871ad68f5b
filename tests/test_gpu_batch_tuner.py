"""The batch autotuner times the instance schedule as a step runs it."""
import numpy as np
import pytest

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


def test_tuned_stage_time_is_that_of_a_step(gpu):
    """Instances of 4^3 to 16^3 elements: a step forks and joins the streams once. With a join after every stage,
    where all instances wait for the slowest one, the reported stage time was 6 to 9 % above a step's; bound 4 %
    (medians of five)."""
    inst = []
    for k, (n, N) in enumerate([(16, 3), (4, 3), (10, 4), (6, 3), (4, 4), (12, 3)]):
        s = nsk.Solver(3, (n,) * 3, N)
        s.set_params(kappa=1e-3, alpha=100.0, beta=1e-2, mu=1e-2)
        g = np.random.Generator(np.random.PCG64(k))
        rho = 1.0 + 1e-3 * g.standard_normal(s.shape[1:])
        s.set_state(np.stack([rho] + [0.0 * rho] * 3 + [rho]))
        inst.append(s)
    b = nsk.Batch(inst)
    b.step(2, cfl=0.1)
    tuned = []
    for _ in range(5):
        _, _, persistent, ms = b.autotune()
        tuned.append(ms)
    assert persistent == nsk.Batch.INSTANCES
    b.step(2)
    stage = min(b.step(10, timings=True)) / 5
    assert np.median(tuned) <= 1.04 * stage, (tuned, stage)
    b.close()
    for s in inst:
        s.close()

"""The benchmark's sequential arm of a batch steps every instance under the schedule the batch runs."""
import sys
from pathlib import Path

import pytest

sys.path.insert(0, str(Path(__file__).resolve().parent.parent))
import bench  # noqa: E402


class _Context:
    """As nsk_set_schedule: a context has schedules 0 to 4."""

    def __init__(self):
        self.schedule = (128, 4)

    def set_schedule(self, tpb, fused):
        if not 0 <= fused <= 4:
            raise ValueError(fused)
        self.schedule = (tpb, fused)


@pytest.mark.parametrize("fused", [0, 1, 2, 4, 5])
def test_solo_schedule_of_a_batch_instance(fused):
    s = _Context()
    bench.solo_schedule(s, 256, fused)
    assert s.schedule == ((128, 4) if fused == 5 else (256, fused))

"""The clock of the kernels' bounded waits, replayed on the host: time in which the GPU is with another program (long gaps
between two readings of its timer) must not run a wait out, time spent waiting must."""
import pytest

from paper_2309_13307_b200 import binding

MS = 1_000_000


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


def test_time_away_does_not_run_a_wait_out():
    # a reading every 20 us; the GPU is away for 150 ms after the third and for ten minutes after the tenth
    readings, now = [], 5 * MS
    for i in range(1000):
        readings.append(now)
        now += 150 * MS if i == 2 else 600_000 * MS if i == 9 else 20_000
    assert binding.core_debug_wait_clock(readings, 100 * MS) == -1


@pytest.mark.parametrize("step", [20_000, 333_333, MS])
def test_time_spent_waiting_does(step):
    readings = [7 + step * i for i in range(6000)]
    at = binding.core_debug_wait_clock(readings, 100 * MS)
    assert (at - 1) * step < 100 * MS <= at * step


def test_every_wait_ends():
    # however far apart the readings are: each counts at least something, 100 of them make 100 ms
    assert binding.core_debug_wait_clock([i * 3_600_000 * MS for i in range(101)], 100 * MS) == 100

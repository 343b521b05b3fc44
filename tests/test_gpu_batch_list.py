"""What a batch does on the host before its launch."""
import time

import numpy as np
import pytest

from paper_2604_21128_gb300 import inputs, qla

pytestmark = pytest.mark.gpu


def step_time(count, rows):
    """Best wall time of a step of `count` lattices of 128 x 8."""
    n = np.full((8, 128), 1.5)
    q0 = inputs.random_state(128, 8, seed=1, planes=3)
    with qla.Batch([(128, 8)] * count, 1.0, "fp32", te_only=True) as b:
        b.set_tuning(0, rows)
        for k in range(count):
            g = b.instance(k)
            g.set_medium(n)
            g.set_state(q0)
        b.step(2)
        best = 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            b.step(1)
            best = min(best, time.perf_counter() - t0)
    return best


def test_choosing_the_row_count_is_a_small_part_of_a_step():
    # the choice looks at every lattice at most eight times (rows 128 to 16);
    # a step with rows given visits each several times as well (generations,
    # geometry, instance records).  Choosing anew for each lattice instead
    # would look at up to 8 x 1024 of them 1024 times.
    given, chosen = step_time(1024, 32), step_time(1024, 0)
    print("batch step: rows given %.2f ms, chosen %.2f ms" % (1e3 * given, 1e3 * chosen))
    assert chosen < 8 * given

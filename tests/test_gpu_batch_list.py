"""What a batch does on the host before its launch: the unit list that it keeps
between calls, and the cost of choosing its row count."""
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


def test_kept_unit_list_follows_media_and_tunings():
    """Calls that keep the list, calls after one instance's medium has changed (a
    plateau where there was none and the other way round) and calls under
    another tiling: every instance as on its own, bit for bit."""
    sizes = [(512, 96), (640, 72), (256, 128)]
    flat = [np.full((ny, nx), 2.0) for nx, ny in sizes]
    rough = [inputs.random_medium(nx, ny, seed=nx, lo=1.0, hi=2.5) for nx, ny in sizes]
    q0 = [inputs.random_state(nx, ny, seed=ny, planes=3) for nx, ny in sizes]
    # (instance whose medium changes, its medium, tuning) before each call of 3 steps
    calls = [(None, None, None), (1, rough[1], None), (1, flat[1], None), (2, flat[2], None),
             (None, None, (1, 64)), (None, None, (0, 0)), (0, rough[0], None)]
    with qla.Batch(sizes, 1.0, "fp32", te_only=True) as b:
        media = [flat[0], flat[1], rough[2]]
        for k in range(3):
            b.instance(k).set_medium(media[k])
            b.instance(k).set_state(q0[k])
        for k, n, tuning in calls:
            if k is not None:
                b.instance(k).set_medium(n)
            if tuning:
                b.set_tuning(*tuning)
            b.step(3)
        got = [b.instance(k).get_state() for k in range(3)]
    for k, (nx, ny) in enumerate(sizes):
        with qla.Grid(nx, ny, 1.0, "fp32", te_only=True) as g:
            g.set_step_kernel("tile")
            g.set_medium(media[k])
            g.set_state(q0[k])
            for j, n, _ in calls:
                if j == k:
                    g.set_medium(n)
                g.step(3)
            assert np.array_equal(got[k], g.get_state()), k

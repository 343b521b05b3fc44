"""The plateau split of six-plane FP32 steps (the two decoupled triples of a
unit list in one launch) against the unsplit march, bit for bit, at segment
heights that leave ragged ends, for each potential reading it takes."""
import numpy as np
import pytest

from paper_2604_21128_gb300 import inputs, qla

pytestmark = pytest.mark.gpu


# the last value: whether any window lies on one plateau (else the step is the
# unsplit march)
@pytest.mark.parametrize("nx,ny,rows,potential,split",
                         [(512, 200, 16, "rotation", True), (364, 130, 28, "rotation", False),
                          (1024, 90, 64, "literal", True), (128, 77, 20, "none", False)])
def test_six_plane_split_agrees_bitwise(nx, ny, rows, potential, split):
    n = np.full((ny, nx), 2.0)
    n[:, : nx // 3] = 1.0
    n[-20:, -30:] = inputs.random_medium(30, 20, seed=5, lo=1.2, hi=2.8)
    q0 = inputs.random_state(nx, ny, seed=nx + rows)
    out = {}
    for kernel in ("march", "march_plain"):
        with qla.Grid(nx, ny, 1.0, "fp32", potential=potential) as g:
            g.set_step_kernel(kernel)
            g.set_march_tuning(0, rows)
            g.set_medium(n)
            g.set_state(q0)
            g.step(6)
            out[kernel] = g.get_state(), g.energy(), g.march_plan
    assert (out["march"][2][1] > 0) == split and out["march_plain"][2] == (0, 0, 0)
    assert np.array_equal(out["march"][0], out["march_plain"][0])
    assert out["march"][1] == out["march_plain"][1]


@pytest.mark.parametrize("kernel,rows,split", [("auto", 64, False), ("march", 64, True),
                                               ("march", 12, False)])
def test_rows_force_the_split_only_where_it_is_asked_for(kernel, rows, split):
    """A lattice below the split's line (2048 x 1024): an automatic context with
    rows set keeps the unsplit march, as does any with rows the units cannot
    have; all give the same bits."""
    nx, ny = 2048, 1024
    n = np.full((ny, nx), 2.0)
    n[:, : nx // 3] = 1.0
    q0 = inputs.random_state(nx, ny, seed=rows)
    out = []
    for k, r in ((kernel, rows), ("march_plain", 0)):
        with qla.Grid(nx, ny, 1.0, "fp32") as g:
            g.set_step_kernel(k)
            g.set_march_tuning(0, r)
            g.set_medium(n)
            g.set_state(q0)
            g.step(3)
            out.append((g.march_plan[1] > 0, g.get_state()))
    assert out[0][0] == split and not out[1][0]
    assert np.array_equal(out[0][1], out[1][1])


def test_six_plane_split_without_a_potential():
    test_six_plane_split_agrees_bitwise(512, 77, 20, "none", True)


def test_automatic_six_plane_split():
    """A lattice just above the line of split6_segment, at the height it picks."""
    import torch
    nx, ny = 3400, 3376
    n = np.full((ny, nx), 2.0)
    n[:, : nx // 3] = 1.0
    n[-60:, -90:] = inputs.random_medium(90, 60, seed=5, lo=1.2, hi=2.8)
    q0 = inputs.random_state(nx, ny, seed=12)
    out = []
    for kernel in ("auto", "march_plain"):
        with qla.Grid(nx, ny, 1.0, "fp32") as g:
            g.set_step_kernel(kernel)
            g.set_medium(n)
            g.set_state(q0)
            g.step(3)
            out.append((g.march_plan[1], g.pack_box(0, 0, nx, ny)))
    assert out[0][0] > 0 and out[1][0] == 0
    assert torch.equal(out[0][1], out[1][1])

"""Resident-tile launches (all steps of a qla_step call on a small lattice in
one launch of the tile kernel, tiles waiting for their neighbours) against one
tile launch per step: the same bits at the edges of the tile sizes, for every
potential reading and medium, and a wait that runs out is reported."""
import time

import numpy as np
import pytest

from paper_2604_21128_gb300 import inputs, qla

pytestmark = pytest.mark.gpu

# one tile, one tile and a site, tiles of 12 and 13, long and thin, many tiles
SHAPES = [(5, 7), (24, 24), (25, 24), (47, 49), (130, 9), (33, 260), (256, 251)]


def run(shape, kernel, calls, precision="fp32", te=True, potential="rotation", tensor=False):
    nx, ny = shape
    n = inputs.random_medium(nx, ny, seed=nx + 7 * ny, lo=1.0, hi=2.5)
    n[: ny // 2] = 2.0                      # shared records next to own ones
    with qla.Grid(nx, ny, 1.0, precision, te_only=te, potential=potential, tensor=tensor) as g:
        g.set_step_kernel(kernel)
        g.set_medium(np.stack([n, 1.1 * n, 1.2 * n]) if tensor else n)
        g.set_state(inputs.random_state(nx, ny, seed=nx, planes=3 if te else 6))
        before = g.launches
        for k in calls:
            g.step(k)
        return g.launches - before, g.get_state(), g.energy()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("te", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_resident_tiles_agree_bitwise(shape, te, precision):
    a = run(shape, "auto", (4, 1, 6), precision, te)
    b = run(shape, "tile", (11,), precision, te)
    assert a[0] == 3 and b[0] == 11
    assert np.array_equal(a[1], b[1]) and a[2] == b[2]


@pytest.mark.parametrize("shape,te,kw", [((300, 301), True, {}), ((512, 500), True, {}),
                                         ((700, 650), True, dict(potential="literal")),
                                         ((1500, 120), True, {}), ((400, 390), False, {}),
                                         ((330, 280), False, dict(tensor=True)),
                                         ((333, 290), False, dict(potential="lcu"))])
def test_several_resident_tiles_per_sm(shape, te, kw):
    """More tiles than SMs (eight warps each), up to six per SM."""
    a = run(shape, "auto", (4, 1, 6), "fp32", te, **kw)
    b = run(shape, "tile", (11,), "fp32", te, **kw)
    assert a[0] == 3 and b[0] == 11
    assert np.array_equal(a[1], b[1]) and a[2] == b[2]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kw", [dict(potential="literal"), dict(potential="none"),
                                dict(potential="lcu"), dict(te=False, potential="lcu"),
                                dict(te=False, tensor=True),
                                dict(te=False, tensor=True, potential="lcu")])
def test_resident_tiles_of_every_reading(kw, precision):
    a = run((61, 50), "auto", (5,), precision, **kw)
    b = run((61, 50), "tile", (5,), precision, **kw)
    assert a[0] == 1 and b[0] == 5
    assert np.array_equal(a[1], b[1]) and a[2] == b[2]


def test_tile_wait_runs_out_without_fault():
    """A tile that does not publish a step: its neighbours wait out a short
    limit, every CTA leaves, the next read returns QLA_ETIMEOUT, and with the
    state set again the context steps exactly as before."""
    nx, ny = 96, 72
    n = inputs.random_medium(nx, ny, seed=3)
    q0 = inputs.random_state(nx, ny, seed=4)
    out = []
    with qla.Grid(nx, ny, 1.0, "fp64") as g:
        g.set_medium(n)
        for withhold in (3, -1):
            g.set_state(q0)
            g.debug_flow(budget_cycles=2_000_000 if withhold >= 0 else 0, withhold_unit=withhold)
            t0 = time.perf_counter()
            g.step(6)
            if withhold >= 0:
                with pytest.raises(qla.QLAError) as e:
                    g.energy()
                assert e.value.status == 5     # QLA_ETIMEOUT
                assert time.perf_counter() - t0 < 30.0
        out.append(g.get_state())
    with qla.Grid(nx, ny, 1.0, "fp64") as g:
        g.set_step_kernel("tile")
        g.set_medium(n)
        g.set_state(q0)
        g.step(6)
        out.append(g.get_state())
    assert np.array_equal(out[0], out[1])


def test_captured_steps_report_their_waits():
    """Steps captured into graphs: a replay whose wait runs out is reported by
    the read after it, each time; another graph of the same context, captured
    before any read, then runs as it should."""
    import torch
    nx, ny = 96, 72
    n = inputs.random_medium(nx, ny, seed=3)
    q0 = inputs.random_state(nx, ny, seed=4)
    stream = torch.cuda.Stream()
    with qla.Grid(nx, ny, 1.0, "fp64", stream=stream) as g:
        def start():
            g.set_state(q0)
            g.step(2)
        g.set_medium(n)
        start()
        graphs = []
        for withhold in (3, -1):
            g.debug_flow(budget_cycles=2_000_000 if withhold >= 0 else 0, withhold_unit=withhold)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                g.step(6)
            graphs.append(graph)
        g.energy()
        for _ in range(2):
            with torch.cuda.stream(stream):
                graphs[0].replay()
            with pytest.raises(qla.QLAError) as e:
                g.energy()
            assert e.value.status == 5     # QLA_ETIMEOUT
            start()
        g.energy()
        with torch.cuda.stream(stream):
            graphs[1].replay()
        got = g.get_state()
        del graphs
    with qla.Grid(nx, ny, 1.0, "fp64") as g:
        g.set_step_kernel("tile")
        g.set_medium(n)
        g.set_state(q0)
        g.step(8)
        assert np.array_equal(got, g.get_state())


@pytest.mark.parametrize("calls", [(1, 2, 3), (8,)])
def test_short_calls_take_resident_tiles_and_a_plan_is_described(calls):
    """512^2 E_z lattices: calls of any length are one launch each, and the plan
    of the marching step is described when asked for."""
    nx = ny = 512
    n = np.full((ny, nx), 2.0)
    n[:, : nx // 3] = 1.0
    q0 = inputs.random_state(nx, ny, seed=9, planes=3)
    out = {}
    for kernel in ("auto", "tile", "march"):
        with qla.Grid(nx, ny, 1.0, "fp32", te_only=True) as g:
            g.set_step_kernel(kernel)
            g.set_medium(n)
            g.set_state(q0)
            assert g.march_plan == (0, 0, 0)       # no step yet
            before = g.launches
            for k in calls:
                g.step(k)
            out[kernel] = g.launches - before, g.get_state(), g.march_plan
            g.set_medium(n)
            assert g.march_plan == (0, 0, 0)
    assert out["auto"][0] == len(calls) and out["tile"][0] == sum(calls)
    assert np.array_equal(out["auto"][1], out["tile"][1])
    assert np.array_equal(out["auto"][1], out["march"][1])
    assert out["auto"][2] == out["march"][2] and out["auto"][2][1] > 0
    assert out["tile"][2] == (0, 0, 0)


@pytest.mark.parametrize("precision,te,lane_cols,rows",
                         [("fp32", True, 1, 0), ("fp32", True, 0, 32), ("fp64", True, 0, 16),
                          ("fp32", False, 0, 8)])
def test_a_tuning_takes_the_marching_kernel(precision, te, lane_cols, rows):
    nx, ny = 128, 96
    n = inputs.random_medium(nx, ny, seed=5, lo=1.0, hi=2.5)
    q0 = inputs.random_state(nx, ny, seed=6, planes=3 if te else 6)
    out = {}
    for kernel in ("auto", "march_step" if precision == "fp32" and te else "march"):
        with qla.Grid(nx, ny, 1.0, precision, te_only=te) as g:
            g.set_step_kernel(kernel)
            g.set_march_tuning(lane_cols, rows)
            g.set_medium(n)
            g.set_state(q0)
            before = g.launches
            g.step(7)
            out[kernel] = g.launches - before, g.get_state()
            g.set_march_tuning()                   # resident tiles again
            before = g.launches
            g.step(5)
            if kernel == "auto":
                assert g.launches - before == 1
    (a, sa), (b, sb) = out.values()
    assert a == b == 7 and np.array_equal(sa, sb)

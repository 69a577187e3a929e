"""The cost of advection steps on large grids, where a sweep should be little
more than moving each cell once."""
import time

import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = pytest.mark.gpu


def _open(n):
    p = inputs.c1_advection(n)
    p.polygons, p.moving = [], []
    return p


def _step_ms(probs, precision, steps):
    from paper_1711_11361_gb300 import mb
    sim = mb.Sim(probs, precision)
    best = 1e30
    for _ in range(6):
        t0 = time.perf_counter()
        sim.run(steps)
        sim.sync()
        best = min(best, time.perf_counter() - t0)
    sim.close()
    return 1e3 * best / steps


def test_constant_speeds_take_no_atomic_per_warp():
    """4096 x 4096 cells in FP32: 0.99 ms per step with a pair of atomics for every warp of 30 cells in the last sweep,
    0.59 without."""
    assert _step_ms(_open(4096), 1, 20) <= 0.8


@pytest.mark.parametrize("precision", [0, 1])
def test_no_body_no_second_launch(precision):
    """A batch without a body is swept by one launch per direction: no more kernels than with the overlap off."""
    from paper_1711_11361_gb300 import mb
    sim = mb.Sim([_open(64), _open(96)], precision)
    kernels = []
    for on in (True, False):
        sim.set_overlap(on)
        sim.run(4)
        sim.sync()
        kernels.append(sim.graph_kernels())
    assert kernels[0] == kernels[1], kernels
    sim.close()


def test_several_units_per_warp():
    """4096 x 4096 cells in FP32: 0.47 ms per step with a unit of 30 cells per warp, 0.24 with four (0.24 with a warp
    per row or segment of rows)."""
    assert _step_ms(_open(4096), 1, 20) <= 0.36


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("nx,ny", [(119, 8), (120, 31), (121, 30), (8, 257), (33, 61), (63, 29), (240, 90)])
def test_wide_units_give_the_same_bits(nx, ny, periodic, precision):
    """A small grid around the channel's walls in a batch large enough for four units per warp, and alone: the units'
    ends lie elsewhere, the arithmetic per cell is the same."""
    from paper_1711_11361_gb300 import mb
    p = inputs.c1_advection(64)
    p.nx, p.ny = nx, ny
    if not periodic:
        p.bc = (inputs.TRANSMISSIVE, inputs.TRANSMISSIVE, inputs.REFLECTIVE, inputs.TRANSMISSIVE)
    rng = np.random.default_rng(nx + ny)
    p.Q0 = rng.uniform(0.5, 1.5, (1, ny, nx))
    big = _open(1500)
    alone, batch = mb.Sim(p, precision), mb.Sim([p, big, p], precision)
    for k in range(3):
        dt = alone.step(0.0, report=True)[0]
        batch.step(float(dt))
    want = alone.read_state(0, alpha=True)
    for k in (0, 2):
        got = batch.read_state(k, alpha=True)
        assert np.array_equal(got["Q"], want["Q"], equal_nan=True) and np.array_equal(got["alpha"], want["alpha"])
    assert np.any(want["alpha"] == 0.0) and np.all(np.isfinite(want["Q"][:, want["alpha"] > 0]))
    alone.close()
    batch.close()

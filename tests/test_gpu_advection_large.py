"""The cost of advection steps on large grids, where a sweep should be little
more than moving each cell once."""
import time

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

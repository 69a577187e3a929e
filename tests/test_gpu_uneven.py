"""Batches of very uneven grids: the kernels numbered by blocks of cells find
their instance (blocks of 2048 cells, the search looks at 32 instances at a
time), and a large grid among small ones costs what its cells cost."""
import time

import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [(8, 8), (45, 45), (46, 45), (64, 32), (64, 33), (300, 9), (8, 257), (129, 128)]


def _tube(nx, ny, axisym=True, seed=0):
    p = inputs.Problem("tube", nx, ny, 0.0, 0.0, 1.0, 1.0, axisym=axisym,
                       bc=(inputs.TRANSMISSIVE, inputs.TRANSMISSIVE, inputs.REFLECTIVE, inputs.TRANSMISSIVE))
    rng = np.random.default_rng(seed)
    y = (np.arange(ny) + 0.5)[:, None] / ny
    p.Q0 = inputs.conserved(1.0 + 0.1 * rng.random((ny, nx)), 0.1, 0.3 * y * np.ones((1, nx)), 1.0 + 0.1 * rng.random((ny, nx)))
    return p


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [1, 31, 32, 33, 65, 1030])
def test_axisymmetric_source_of_every_instance(count, precision):
    from paper_1711_11361_gb300 import mb
    # (every third one without the source)
    kinds = [_tube(nx, ny, k % 3 != 2, k) for k, (nx, ny) in enumerate(SIZES)]
    order = np.random.default_rng(count).integers(0, len(SIZES), count)
    sim = mb.Sim([kinds[k] for k in order], precision)
    sim.step(1e-3)
    got = sim.read_states()[0]
    for k in set(order.tolist()):
        alone = mb.Sim(kinds[k], precision)
        alone.step(1e-3)
        want = alone.read_state(0)["Q"]
        alone.close()
        for at in np.where(order == k)[0]:
            assert np.array_equal(got[at], want), (k, at)
    sim.close()


def _best(f, n=5):
    f()
    t = []
    for _ in range(n):
        t0 = time.perf_counter()
        f()
        t.append(time.perf_counter() - t0)
    return min(t)


def test_cost_of_the_source_in_an_uneven_batch():
    """One grid of 4096 x 4096 cells and 63 of 128 x 128: the source moves every state once more, after two sweeps
    that do so too, so a step with it takes less than twice one without (1.3 times; 4 times where every instance
    got as many CTAs as the largest)."""
    from paper_1711_11361_gb300 import mb
    t = []
    for axisym in (False, True):
        sim = mb.Sim([_tube(4096, 4096, axisym)] + [_tube(128, 128, axisym)] * 63, mb.FP32)

        def steps():
            sim.run(10, 1e-6)
            sim.sync()

        t.append(_best(steps))
        sim.close()
    assert t[1] <= 2.0 * t[0], t

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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [2, 31, 32, 33, 65, 1030])
def test_states_of_every_instance(count, precision):
    """Every instance's own state in and out, some left out of the read; the first step from each one's own speeds."""
    from paper_1711_11361_gb300 import mb
    kinds = [_tube(nx, ny, False, k) for k, (nx, ny) in enumerate(SIZES)]
    order = np.random.default_rng(count).integers(0, len(SIZES), count)
    scale = 1.0 + np.arange(count) % 64 / 64.0
    states = [kinds[k].Q0 * s for k, s in zip(order, scale)]
    dtype = np.float32 if precision else np.float64
    sim = mb.Sim([kinds[k] for k in order], precision, write_initial=False)
    sim.write_states(states)
    out = [np.full(q.shape, -7.0) for q in states]
    ptrs = sim._ptrs(out)
    for at in range(0, count, 3):
        ptrs[at] = None
    clk = np.empty((count, 4))
    sim._check(mb.lib.mb_read_states(sim._h, ptrs, mb._dp(clk)))
    for at in range(count):
        assert np.array_equal(out[at], np.full(out[at].shape, -7.0) if at % 3 == 0 else states[at].astype(dtype)), at
    got = sim.step(0.0, report=True)
    sim.close()
    for k in set(order.tolist()):
        q = [states[at].astype(dtype).astype(np.float64) for at in np.where(order == k)[0]]
        for at, x in zip(np.where(order == k)[0], q):
            p = kinds[k]
            c = np.sqrt(p.gamma * (p.gamma - 1.0) * (x[3] - 0.5 * (x[1] ** 2 + x[2] ** 2) / x[0]) / x[0])
            want = p.cfl * min(p.dx / np.max(np.abs(x[1] / x[0]) + c), p.dy / np.max(np.abs(x[2] / x[0]) + c))
            assert abs(got[at] - want) <= 1e-14 * want, at


def test_cost_of_state_copies_in_an_uneven_batch():
    """Writing and reading 2000 grids of 8 x 8 cells and one of 4096 x 4096 takes about as long as the small ones and
    the large one apart (well beyond the bar where every instance got as many CTAs as the largest)."""
    import torch

    from paper_1711_11361_gb300 import mb

    def cost(shapes):
        probs = [_tube(8, 8, False) for _ in range(shapes.count(8))]
        probs += [inputs.Problem("large", 4096, 4096, 0.0, 0.0, 1.0, 1.0) for _ in range(shapes.count(4096))]
        bufs = [torch.empty((4, p.ny, p.nx), pin_memory=True) for p in probs]
        for b in bufs:
            b[:] = torch.tensor([1.0, 0.1, 0.2, 2.5])[:, None, None]
        sim = mb.Sim(probs, mb.FP32, write_initial=False)
        at = [b.data_ptr() for b in bufs]
        t = _best(lambda: (sim.write_states(at, dtype=np.float32), sim.read_states(out=at, dtype=np.float32)))
        sim.close()
        return t

    both, apart = cost([8] * 2000 + [4096]), cost([8] * 2001) + cost([4096, 8])
    assert both <= 1.5 * apart, (both, apart)

"""The positivity test of an updated cell in units of mass near the ends of
FP32's range: the arithmetic scales exactly by powers of two, so a sweep over a
state with a few non-physical cells (2 rho E one per cent below m^2) merges the
same cells and leaves the same bits, times the scale, as in ordinary units."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

POWERS = [-74, -62, -40, 40, 62]   # (62: products of energies pass 1e38)


def _momenta(shape, parts, rng):
    # every square is 0.2, signs vary: the cells' speeds differ
    return [np.sqrt(0.2) * rng.choice([-1.0, 1.0], shape) for _ in range(parts)]


@pytest.mark.parametrize("power", POWERS)
def test_two_dimensions(power):
    from paper_1711_11361_gb300 import mb
    rng, shape = np.random.default_rng(5), (40, 70)
    m = _momenta(shape, 2, rng)
    E = np.full(shape, 1.0)
    E[rng.integers(0, 40, 6), rng.integers(0, 70, 6)] = 0.99 * 0.5 * 0.4
    p = inputs.Problem("units", 70, 40, 0.0, 0.0, 1.0, 1.0, bc=(inputs.PERIODIC,) * 4)
    p.Q0 = np.stack([np.ones(shape), *m, E])
    for d in (0, 1):
        out = []
        for s in (1.0, 2.0 ** power):
            sim = mb.Sim(p, mb.FP64, write_initial=False)
            sim.write_state(0, p.Q0 * s)
            sim.sweep(d, 1e-9)
            out.append((sim.read_state(0)["Q"] / s, sim.diagnostics(0)["mixed"]))
            sim.close()
        assert out[0][1] > 0 and out[1][1] == out[0][1]
        assert np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("power", POWERS)
def test_three_dimensions(power):
    from paper_1711_11361_gb300 import mb3
    rng, shape = np.random.default_rng(6), (9, 11, 33)
    m = _momenta(shape, 3, rng)
    E = np.full(shape, 1.0)
    E[rng.integers(0, 9, 5), rng.integers(0, 11, 5), rng.integers(0, 33, 5)] = 0.99 * 0.5 * 0.6
    p = inputs.Problem3("units", 33, 11, 9, bc=(inputs.PERIODIC,) * 6)
    Q = np.stack([np.ones(shape), *m, E])
    for d in range(3):
        out = []
        for s in (1.0, 2.0 ** power):
            sim = mb3.Sim3(p, write_initial=False)
            sim.write_state(Q * s)
            sim.sweep(d, 1e-9)
            out.append((sim.read_state()["Q"] / s, sim.last_sweep()[1]))
            sim.close()
        assert out[0][1] > 0 and out[1][1] == out[0][1]
        assert np.array_equal(out[0][0], out[1][0])

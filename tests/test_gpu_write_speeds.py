"""The first step's dt of a written state, where the screening of its wave
speeds divides: one, two or three distinct states per block of 2048 cells,
speeds that tie between different states, random states, a low pressure that
the FP32 screen does not trust; grids of just under, just over and several
blocks, both precisions.  Against the speeds of every cell in numpy: 1e-14
relative, the bound of the CFL parity tests (a few roundings)."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def _state(kind, shape, rng):
    X = np.broadcast_to(np.arange(shape[1])[None, :], shape)
    one = np.ones(shape)
    if kind == "uniform":
        return inputs.conserved(one, 0.3, -0.2, one)
    if kind == "two":
        left = X < shape[1] // 3
        return inputs.conserved(np.where(left, 1.0, 2.0), np.where(left, 0.3, -0.4), 0.1, np.where(left, 1.0, 2.5))
    if kind == "three":
        k = X % 3
        return inputs.conserved(1.0 + k, 0.1 * k, -0.3 * k, 1.0 + 0.5 * k)
    if kind == "ties":   # scaling keeps velocity and sound speed
        return inputs.conserved(one, 0.3, -0.2, one) * (1.0 + 0.01 * np.sin(0.1 * X))
    p = np.full(shape, 1e-3) if kind == "low pressure" else rng.uniform(0.2, 3.0, shape)
    return inputs.conserved(rng.uniform(0.2, 3.0, shape), rng.uniform(-2, 2, shape), rng.uniform(-2, 2, shape), p)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["uniform", "two", "three", "ties", "random", "low pressure"])
@pytest.mark.parametrize("nx,ny", [(23, 89), (32, 64), (41, 50), (131, 77)])
def test_first_dt(nx, ny, kind, precision):
    from paper_1711_11361_gb300 import mb
    p = inputs.Problem("speeds", nx, ny, 0.0, 0.0, 1.0, 1.3, cfl=0.4)
    p.Q0 = _state(kind, (ny, nx), np.random.default_rng(nx))
    q = (p.Q0.astype(np.float32) if precision else p.Q0).astype(np.float64)
    c = np.sqrt(p.gamma * (p.gamma - 1.0) * (q[3] - 0.5 * (q[1] ** 2 + q[2] ** 2) / q[0]) / q[0])
    want = p.cfl * min(p.dx / np.max(np.abs(q[1] / q[0]) + c), p.dy / np.max(np.abs(q[2] / q[0]) + c))
    for sim in (mb.Sim(p, precision), mb.Sim([p, p], precision)):
        got = sim.step(0.0, report=True)
        assert np.all(np.abs(got - want) <= 1e-14 * want)
        sim.close()

"""mb_write_state's listed cells: numbers of tied states per block of 2048 cells
on both sides of a warp's 32, states that take turns along a row, cells that a
body covers (their host values are no numbers), rows shorter and longer than a
CTA's 256 threads, both precisions.  The first step against the speeds of every
fluid cell in numpy to 1e-14 (the bound of the CFL parity tests), the state read
back bit for bit."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def _check(mb, p, precision, fluid=None):
    q = (p.Q0.astype(np.float32) if precision else p.Q0).astype(np.float64)
    fluid = np.ones(q[0].shape, bool) if fluid is None else fluid
    c = np.sqrt(p.gamma * (p.gamma - 1.0) * (q[3] - 0.5 * (q[1] ** 2 + q[2] ** 2) / q[0]) / q[0])
    want = p.cfl * min(p.dx / np.max((np.abs(q[1] / q[0]) + c)[fluid]), p.dy / np.max((np.abs(q[2] / q[0]) + c)[fluid]))
    for probs in (p, [p, p]):
        sim = mb.Sim(probs, precision)
        back = sim.read_state(0)["Q"]
        assert np.array_equal(back[:, fluid], q[:, fluid]) and np.all(np.isnan(back[:, ~fluid]))
        assert np.all(np.abs(sim.step(0.0, report=True) - want) <= 1e-14 * want)
        sim.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ties", [1, 2, 31, 32, 33, 64, 65, 256, 257, 2048])
@pytest.mark.parametrize("nx,ny", [(8, 300), (256, 9), (257, 17), (700, 8)])
def test_tied_states(nx, ny, ties, precision):
    from paper_1711_11361_gb300 import mb
    p = inputs.Problem("ties", nx, ny, 0.0, 0.0, 1.0, 1.3, cfl=0.4)
    n, rng = nx * ny, np.random.default_rng(ties)
    # in each block of 2048 cells `ties` distinct states, equal speeds to a rounding (scaled by powers of two and by
    # short fractions), in turns; the rest in one slower state
    e = np.arange(n)
    scale = 1.0 + (e % 2048 % ties) / 4096.0
    slow = (e % 2048) * 1.0 >= max(ties, 1) * max(1, 2048 // ties // 2)
    q = inputs.conserved(np.ones(n), 0.3, -0.2, np.ones(n)) * scale
    q[:, slow] = inputs.conserved(np.ones(1), 0.1, 0.1, np.full(1, 0.5))
    if rng.random() < 0.5:
        q = q[:, ::-1]
    p.Q0 = np.ascontiguousarray(q.reshape(4, ny, nx))
    _check(mb, p, precision)


@pytest.mark.parametrize("precision", [0, 1])
def test_covered_cells(precision):
    from paper_1711_11361_gb300 import mb
    p = inputs.c2_cylinder(96)
    sim = mb.Sim(p, precision)
    fluid = sim.read_state(0, alpha=True)["alpha"] > 0
    sim.close()
    assert np.sum(~fluid) > 20
    rng = np.random.default_rng(1)
    p.Q0 = p.Q0 * (1.0 + 0.01 * rng.integers(0, 3, p.Q0.shape[1:]))
    p.Q0[:, ~fluid] = np.nan
    _check(mb, p, precision, fluid)

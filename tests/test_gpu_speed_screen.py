"""Wave speeds behind the CFL step where their FP32 screen is least accurate:
cells whose speeds agree to 1e-7, with a pressure just above the screen's bound
(and a tenth of the energy), the largest in a cell whose FP32 speed comes out
lowest; adiabatic exponents from 1.1 to 20; and units of mass that put the
momenta's squares outside FP32's range.  A written state's first step, the step
after an update and the three-dimensional CFL step against the speeds of every
cell in numpy: 1e-12 relative (a few FP64 roundings, amplified up to 200
times by 2 E - m^2 / rho, are below 1e-13; the fastest cell leads by 1e-9)."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

GAMMAS = [1.1, 1.4, 5.0 / 3.0, 3.0, 7.0, 20.0]
BAR = 1e-12


def speeds(q, g):
    """|u| + c of rho, m, E"""
    p = (g - 1.0) * (q[2] - 0.5 * q[1] ** 2 / q[0])
    return np.abs(q[1] / q[0]) + np.sqrt(g * p / q[0])


def screened(q, g):
    """the same in FP32 from inputs cut to 24 bits"""
    x = [(v.view(np.int64) & ~np.int64(0x1fffffff)).view(np.float64).astype(np.float32) for v in q]
    f = np.float32
    ir = f(1) / x[0]
    p = f(g - 1.0) * (x[2] - f(0.5) * x[1] * x[1] * ir)
    return np.abs(x[1] * ir) + np.sqrt(f(g) * p * ir)


def cells(n, g, low, f32, rng):
    """n states (rho, m, E) with |u| + c = 1 to 1e-7; the last one is the fastest, by 1e-9 at least, and of these the
    one whose FP32 speed is least; the others are those whose FP32 speeds are largest.  low: p = 0.1 E, else
    2 E - m^2 / rho = E / 2, both by up to 1% more"""
    pool = 16 * n
    rho = rng.uniform(0.5, 2.0, pool)
    share = (0.2 / (g - 1.0) if low else 0.5) * (1.0 + rng.uniform(1e-4, 1e-2, pool))   # (2 E - m^2 / rho) / E
    share = np.minimum(share, 1.9)
    # E = m^2 / rho / (2 - share), p = (g - 1) / 2 share E
    E1 = rho / (2.0 - share)                                                            # for u = 1
    c1 = np.sqrt(g * 0.5 * (g - 1.0) * share * E1 / rho)
    u = (1.0 + rng.uniform(-1e-7, 1e-7, pool)) / (1.0 + c1)
    q = np.stack([rho, rho * u, E1 * u * u])
    if f32:
        q = q.astype(np.float32).astype(np.float64)
    s, err = speeds(q, g), screened(q, g) / speeds(q, g) - 1.0
    top = np.argmin(np.where(s > np.quantile(s, 0.5), err, 1.0))
    rest = np.where(s < s[top] - 1e-9)[0]
    rest = rest[np.argsort(-err[rest])][:n - 1]
    return np.concatenate([q[:, rng.permutation(rest)], q[:, top:top + 1]], axis=1)


def grid(nx, ny, g, low, f32, seed):
    q = cells(nx * ny, g, low, f32, np.random.default_rng(seed)).reshape(3, ny, nx)
    p = inputs.Problem("speeds", nx, ny, 0.0, 0.0, 1.0, 1.0, cfl=0.4, bc=(inputs.PERIODIC,) * 4)
    p.gamma = g
    p.Q0 = np.stack([q[0], q[1], np.zeros_like(q[0]), q[2]])
    return p


def first_dt(p, q):
    c = np.sqrt(p.gamma * (p.gamma - 1.0) * (q[3] - 0.5 * (q[1] ** 2 + q[2] ** 2) / q[0]) / q[0])
    return p.cfl * min(p.dx / np.max(np.abs(q[1] / q[0]) + c), p.dy / np.max(np.abs(q[2] / q[0]) + c))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("low", [True, False], ids=["tenth", "half"])
@pytest.mark.parametrize("gamma", GAMMAS)
def test_written_state(gamma, low, precision):
    from paper_1711_11361_gb300 import mb
    p = grid(64, 66, gamma, low, precision == 1, 1)
    sim = mb.Sim(p, precision)
    assert abs(sim.step(0.0, report=True)[0] / first_dt(p, p.Q0) - 1.0) <= BAR
    sim.close()


@pytest.mark.parametrize("low", [True, False], ids=["tenth", "half"])
@pytest.mark.parametrize("gamma", GAMMAS)
def test_after_a_step(gamma, low):
    from paper_1711_11361_gb300 import mb
    p = grid(400, 300, gamma, low, False, 2)
    sim = mb.Sim(p, mb.FP64)
    sim.step(1e-16)
    q = sim.read_state(0)["Q"]
    assert abs(sim.step(0.0, report=True)[0] / first_dt(p, q) - 1.0) <= BAR
    sim.close()


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("low", [True, False], ids=["tenth", "half"])
@pytest.mark.parametrize("gamma", GAMMAS)
def test_three_dimensions(gamma, low, axis):
    from paper_1711_11361_gb300 import mb3
    shape = (17, 19, 25)
    q = cells(17 * 19 * 25, gamma, low, False, np.random.default_rng(3)).reshape((3,) + shape)
    p = inputs.Problem3("speeds", 25, 19, 17, bc=(inputs.PERIODIC,) * 6, cfl=0.4)
    p.gamma = gamma
    m = np.zeros((3,) + shape)
    m[axis] = q[1]
    p.Q0 = np.concatenate([q[:1], m, q[2:]])
    c = np.sqrt(gamma * (gamma - 1.0) * (q[2] - 0.5 * q[1] ** 2 / q[0]) / q[0])
    want = p.cfl * min(p.h[a] / np.max(np.abs(m[a] / q[0]) + c) for a in range(3))
    sim = mb3.Sim3(p)
    assert abs(sim.cfl_dt() / want - 1.0) <= BAR
    sim.close()


@pytest.mark.parametrize("scale", [1e-21, 1e-25, 1e20, 1e28], ids=str)
def test_densities_far_from_one(scale):
    """The same cells in other units of mass: a square of a momentum underflows or overflows in FP32."""
    from paper_1711_11361_gb300 import mb, mb3
    p = grid(64, 66, 1.4, True, False, 4)
    p.Q0 *= scale
    p.y1 = 0.2
    # every other row at rest, with the larger speed of sound (0.26 against 0.23, and 0.47 where m^2 is lost), which
    # sets the step along y
    p.Q0[:, ::2] *= np.array([1.0, 0.0, 1.0, 0.3])[:, None, None]
    sim = mb.Sim(p, mb.FP64)
    sim.step(1e-16)
    q = sim.read_state(0)["Q"]
    assert abs(sim.step(0.0, report=True)[0] / first_dt(p, q) - 1.0) <= BAR
    sim.write_state(0, p.Q0)
    assert abs(sim.step(0.0, report=True)[0] / first_dt(p, p.Q0) - 1.0) <= BAR
    sim.close()
    p3 = inputs.Problem3("speeds", 64, 66, 1, hi=(1.0, 0.2, 1.0), bc=(inputs.PERIODIC,) * 6, cfl=0.4)
    p3.Q0 = np.stack([p.Q0[0], p.Q0[1], p.Q0[2], np.zeros_like(p.Q0[0]), p.Q0[3]])[:, None]
    sim3 = mb3.Sim3(p3)
    assert abs(sim3.cfl_dt() / first_dt(p, p.Q0) - 1.0) <= BAR
    sim3.close()

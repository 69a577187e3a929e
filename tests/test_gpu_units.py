"""The scalar bulk kernels (FP64 Euler, advection) at the sizes where their
30-cell units end: grids of one unit, one cell less and more, several units,
every boundary condition, with and without a body.  Against the oracle the
per-sweep bound of the parity tests (contents to 1e-12); the units updated
beside the geometry give the same bits as one launch after it."""
import numpy as np
import pytest

import oracle
from paper_1711_11361_gb300 import inputs

from gpu_util import compare

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

SIZES = [(8, 8), (29, 31), (30, 30), (31, 61), (62, 92), (97, 33)]
SIDES = [(inputs.TRANSMISSIVE,) * 4, (inputs.PERIODIC,) * 4, (inputs.REFLECTIVE,) * 4]


@pytest.fixture(scope="module")
def mb():
    from paper_1711_11361_gb300 import mb as m
    return m


def _problem(nx, ny, bc, equation=inputs.EULER):
    """Smooth state around a moving cylinder (none on the smallest grid) that covers a few cells."""
    r = 2.6 / min(nx, ny)
    polys = [] if min(nx, ny) < 16 else [inputs.cylinder_polygon(0.52, 0.47, r, 1.0 / max(nx, ny))]
    p = inputs.Problem("units", nx, ny, 0.0, 0.0, 1.0, 1.0, bc=bc, equation=equation, adv=(0.8, 0.3), cfl=0.4,
                       polygons=polys, moving=[1] * len(polys), U=(0.4, 0.15), pivot=(0.52, 0.47))
    X, Y = p.cell_centres()
    t = 2.0 * np.pi
    if equation == inputs.ADVECTION:
        p.Q0 = (1.0 + 0.3 * np.sin(t * X) * np.cos(t * Y))[None]
        p.U = (0.0, 0.0)
    else:
        p.Q0 = inputs.conserved(1.0 + 0.2 * np.sin(t * (X + Y)), 0.4 + 0.1 * np.cos(t * Y), 0.15 + 0.1 * np.sin(t * X),
                                1.0 + 0.2 * np.cos(t * X) * np.sin(t * Y))
    return p


@pytest.mark.parametrize("equation", [inputs.EULER, inputs.ADVECTION])
@pytest.mark.parametrize("bc", SIDES, ids=["transmissive", "periodic", "reflective"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_unit_edges(mb, nx, ny, bc, equation):
    prob = _problem(nx, ny, bc, equation)
    orc = oracle.Oracle(prob)
    sim = mb.Sim(prob, mb.FP64)
    dt = orc.cfl_dt()
    for d in (0, 1):
        assert orc.sweep(d, dt) == 0
        sim.sweep(d, dt)
        r = compare(sim, orc)
        assert r["cls"] == 0 and r["contents"] <= 1e-12, (d, r["contents"])


@pytest.mark.parametrize("equation,precision", [(inputs.EULER, 0), (inputs.EULER, 1), (inputs.ADVECTION, 0),
                                                (inputs.ADVECTION, 1)])
def test_far_units_beside_the_geometry(mb, equation, precision):
    probs = [_problem(nx, ny, bc, equation) for nx, ny in SIZES[1:] for bc in SIDES]
    out = []
    for overlap in (True, False):
        sim = mb.Sim(probs, precision)
        sim.set_overlap(overlap)
        sim.run(5)
        out.append([sim.read_state(k)["Q"] for k in range(len(probs))])
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)

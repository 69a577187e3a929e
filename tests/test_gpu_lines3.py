"""The three-dimensional line kernels where their work divides: the cells near
the body against the others, a body against each side (across a periodic one
too), rows and segments one cell over and under a warp's, the shortest axes.
One sweep along each axis from identical input against the oracle (contents
alpha*Q to 1e-12, the one-sweep bound of the three-dimensional parity tests),
and the CFL step; the FP32 option against FP64 by its own bound."""
import math

import numpy as np
import pytest

from oracle import o3
from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

SIDES = {"transmissive": inputs.TRANSMISSIVE, "reflective": inputs.REFLECTIVE, "periodic": inputs.PERIODIC}
# (cells, centre of the body, its half-width in cells), the body's bounding box reaching a side, a corner or the middle
CASES = [((31, 9, 8), (0.5, 0.5, 0.5), 2.2), ((8, 33, 9), (0.45, 0.07, 0.6), 1.7), ((9, 8, 65), (0.5, 0.4, 0.96), 1.9),
         ((61, 7, 6), (0.03, 0.5, 0.5), 1.3), ((30, 32, 3), (0.5, 0.5, 0.5), 4.1), ((2, 64, 29), (0.5, 0.3, 0.3), 0.9),
         ((29, 2, 31), (0.7, 0.5, 0.2), 0.8)]


@pytest.fixture(scope="module")
def mb3():
    from paper_1711_11361_gb300 import mb3 as m
    return m


def _problem(cells, centre, half, side, mode):
    nx, ny, nz = cells
    hi = tuple(n / 10.0 for n in cells)                    # cubic cells of 0.1
    c = np.array([f * h for f, h in zip(centre, hi)]) + 0.0037
    r = 0.1 * half
    nrm = np.concatenate([np.eye(3), -np.eye(3)])
    off = np.concatenate([c + r, r - c])
    bb = tuple(v for a in range(3) for v in (c[a] - r, c[a] + r))
    p = inputs.Problem3("box", nx, ny, nz, hi=hi, normals=nrm, offsets=off, bbox=bb, U=(0.3, -0.2, 0.25), bc=(side,) * 6,
                        uncover_mode=mode, cfl=0.4)
    X, Y, Z = p.cell_centres()
    tx, ty, tz = (2.0 * math.pi / h for h in hi)
    p.Q0 = inputs.conserved3(1 + 0.2 * np.sin(tx * X) * np.cos(ty * Y), 0.3 + 0.1 * np.sin(tz * Z), -0.2 + 0.1 * np.cos(tx * X),
                             0.25 + 0.1 * np.sin(ty * Y), 1 + 0.1 * np.cos(tx * X + tz * Z))
    return p


@pytest.mark.parametrize("mode", [inputs.UNCOVER_DONOR, inputs.UNCOVER_FLUX_GCL], ids=["donor", "gcl"])
@pytest.mark.parametrize("side", list(SIDES))
@pytest.mark.parametrize("cells,centre,half", CASES, ids=["x".join(map(str, c[0])) for c in CASES])
def test_one_sweep_per_axis(mb3, cells, centre, half, side, mode):
    p = _problem(cells, centre, half, SIDES[side], mode)
    for d in range(3):
        orc, sim = o3.Oracle3(p), mb3.Sim3(p)
        dt = orc.cfl_dt()
        assert abs(sim.cfl_dt() - dt) <= 1e-14 * dt
        ro = orc.sweep(d, dt)
        rg = mb3.lib.mb3_sweep(sim._h, d, dt)
        assert rg == ro
        if ro == 0:
            a, b = sim.contents(), orc.contents()
            big = max(np.max(np.abs(b[q])) for q in range(5))
            for q in range(5):
                assert np.max(np.abs(a[q] - b[q])) <= 1e-12 * max(np.max(np.abs(b[q])), 1e-2 * big), (d, q)
        sim.close()


@pytest.mark.parametrize("side", list(SIDES))
def test_fp32_option_at_odd_sizes(mb3, side):
    """The FP32 flux option stays within 1e-4 (relative L1 density, its bar) of the FP64 path."""
    for cells, centre, half in CASES[:5]:
        p = _problem(cells, centre, half, SIDES[side], inputs.UNCOVER_DONOR)
        a, b = mb3.Sim3(p), mb3.Sim3(p, precision=1)
        dt = a.cfl_dt()
        ra, rb = mb3.lib.mb3_sweep(a._h, 0, dt), mb3.lib.mb3_sweep(b._h, 0, dt)
        assert ra == rb
        if ra == 0:
            ca, cb = a.contents(), b.contents()
            assert np.sum(np.abs(ca[0] - cb[0])) <= 1e-4 * np.sum(np.abs(ca[0]))
        a.close()
        b.close()

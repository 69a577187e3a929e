"""Periodic axes of one cell (the quasi-two-dimensional use that mb3_create
accepts) around a body with solid cells: one sweep along each axis from
identical input against the oracle, to 1e-12 of the contents (the one-sweep
bound of the three-dimensional parity tests), in both uncovering modes, and
the FP32 flux option against FP64: every content of every cell within 1e-5 of
its component's scale (some hundred FP32 roundings of 6e-8 on the way from the
state to lam times a flux difference, lam times a wave speed below 1/2)."""
import math

import numpy as np
import pytest

from oracle import o3
from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

CASES = [(24, 20, 1), (20, 1, 24), (1, 24, 20), (33, 1, 1), (1, 1, 40)]


@pytest.fixture(scope="module")
def mb3():
    from paper_1711_11361_gb300 import mb3 as m
    return m


def problem(cells, mode):
    hi = tuple(n / 10.0 for n in cells)
    c = np.array([0.47 * h for h in hi]) + 0.0037
    r = np.array([0.15 if n == 1 else 0.29 for n in cells])      # through a one-cell axis
    nrm = np.concatenate([np.eye(3), -np.eye(3)])
    off = np.concatenate([c + r, r - c])
    bb = tuple(v for a in range(3) for v in (c[a] - r[a], c[a] + r[a]))
    p = inputs.Problem3("thin", *cells, hi=hi, normals=nrm, offsets=off, bbox=bb, U=(0.3, -0.2, 0.25),
                        bc=(inputs.PERIODIC,) * 6, uncover_mode=mode, cfl=0.4)
    X, Y, Z = p.cell_centres()
    tx, ty, tz = (2.0 * math.pi / h for h in hi)
    p.Q0 = inputs.conserved3(1 + 0.2 * np.sin(tx * X) * np.cos(ty * Y), 0.3 + 0.1 * np.sin(tz * Z),
                             -0.2 + 0.1 * np.cos(tx * X), 0.25 + 0.1 * np.sin(ty * Y), 1 + 0.1 * np.cos(tx * X + tz * Z))
    return p


@pytest.mark.parametrize("mode", [inputs.UNCOVER_DONOR, inputs.UNCOVER_FLUX_GCL], ids=["donor", "gcl"])
@pytest.mark.parametrize("cells", CASES, ids=["x".join(map(str, c)) for c in CASES])
def test_sweeps_with_one_cell_axes(mb3, cells, mode):
    p = problem(cells, mode)
    for d in range(3):
        orc, sim, sim32 = o3.Oracle3(p), mb3.Sim3(p), mb3.Sim3(p, precision=1)
        dt = orc.cfl_dt()
        assert orc.sweep(d, dt) == 0
        assert np.sum(orc.alpha() == 0.0) >= 2
        sim.sweep(d, dt)
        sim32.sweep(d, dt)
        a, b, c = sim.contents(), orc.contents(), sim32.contents()
        assert sim.last_sweep()[1] == orc.last_sweep()[1]
        big = max(np.max(np.abs(b[q])) for q in range(5))
        for q in range(5):
            scale = max(np.max(np.abs(b[q])), 1e-2 * big)
            assert np.max(np.abs(a[q] - b[q])) <= 1e-12 * scale, (d, q)
            assert np.max(np.abs(c[q] - a[q])) <= 1e-5 * scale, (d, q)
        for s in (sim, sim32):
            s.close()

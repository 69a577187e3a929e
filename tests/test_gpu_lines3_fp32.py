"""The FP32 flux option of the three-dimensional line kernels where their work
divides (the cases of test_gpu_lines3), along every axis, in both uncovering
modes and on every kind of side: after one sweep each content of each cell lies
within 1e-5 of its component's scale of the FP64 oracle's (some hundred FP32
roundings of 6e-8 on the way from the state to lam times a flux difference, lam
times a wave speed below 1/2), and every sweep succeeds."""
import numpy as np
import pytest

from oracle import o3
from paper_1711_11361_gb300 import inputs
from test_gpu_lines3 import CASES, SIDES, _problem

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("mode", [inputs.UNCOVER_DONOR, inputs.UNCOVER_FLUX_GCL], ids=["donor", "gcl"])
@pytest.mark.parametrize("side", list(SIDES))
@pytest.mark.parametrize("cells,centre,half", CASES, ids=["x".join(map(str, c[0])) for c in CASES])
def test_every_axis(cells, centre, half, side, mode):
    from paper_1711_11361_gb300 import mb3
    p = _problem(cells, centre, half, SIDES[side], mode)
    for d in range(3):
        orc, sim = o3.Oracle3(p), mb3.Sim3(p, precision=1)
        dt = orc.cfl_dt()
        assert orc.sweep(d, dt) == 0
        sim.sweep(d, dt)
        a, b = sim.contents(), orc.contents()
        big = max(np.max(np.abs(b[q])) for q in range(5))
        for q in range(5):
            assert np.max(np.abs(a[q] - b[q])) <= 1e-5 * max(np.max(np.abs(b[q])), 1e-2 * big), (d, q)
        sim.close()

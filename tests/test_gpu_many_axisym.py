"""A batch of more axisymmetric instances than a launch grid's second extent
(65535) holds: created up to it, then added to.  Every one gets the geometric
source (whole numbers of instances apart: the same bits as alone)."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(k):
    p = inputs.Problem("tube", 8, 8, 0.0, 0.0, 1.0, 1.0, axisym=True,
                       bc=(inputs.TRANSMISSIVE, inputs.TRANSMISSIVE, inputs.REFLECTIVE, inputs.TRANSMISSIVE))
    y = (np.arange(8) + 0.5)[:, None] / 8 * np.ones((1, 8))
    p.Q0 = inputs.conserved(1.0 + 0.1 * y, 0.1, 0.3 * y, 1.0 + 0.01 * k + 0.0 * y)
    return p


def test_more_than_65535_instances():
    from paper_1711_11361_gb300 import mb
    kinds = [_problem(k) for k in range(3)]
    sim = mb.Sim([kinds[k % 3] for k in range(65535)], mb.FP64)
    for k in range(2):
        sim.add(kinds[k])
    sim.step(1e-3)
    for k, p in ((0, 0), (40000, 40000 % 3), (65534, 65534 % 3), (65535, 0), (65536, 1)):
        alone = mb.Sim(kinds[p], mb.FP64)
        alone.step(1e-3)
        assert np.array_equal(sim.read_state(k)["Q"], alone.read_state(0)["Q"]), k
        alone.close()
    sim.close()

"""The geometry's edge capacity (384 edges near 16 columns) is the same alone
and in a batch, whatever width the batch gives its geometry groups: what a
large batch refuses, a small one refuses too, and a simulation that runs alone
goes on running when others join it."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def _cylinder(n, vertices):
    p = inputs.c2_cylinder(n)
    q = p.polygons[0]
    c, r = q.mean(0), np.max(np.hypot(*(q - q.mean(0)).T))
    a = 2.0 * np.pi * np.arange(vertices) / vertices
    p.polygons[0] = np.stack([c[0] + r * np.cos(a), c[1] + r * np.sin(a)], 1)
    return p


def _status(sim):
    from paper_1711_11361_gb300 import mb
    try:
        sim.run(2)
        return sim.sync()
    except mb.MBError as e:
        return e.code


# vertices of a cylinder of 60 columns: 16 columns at its sides hold about a third of them
@pytest.mark.parametrize("vertices,status", [(300, 0), (385, 0), (700, 0), (2000, -7)])
@pytest.mark.parametrize("precision", [0, 1])
def test_same_alone_and_in_a_batch(vertices, status, precision):
    from paper_1711_11361_gb300 import mb
    p = _cylinder(300, vertices)
    alone = mb.Sim(p, precision)
    assert _status(alone) == status
    batch = mb.Sim([p] + [inputs.small_case("piston", 128)] * 60, precision)
    assert _status(batch) == status
    if status == 0:
        assert np.array_equal(alone.read_state(0)["Q"], batch.read_state(0)["Q"], equal_nan=True)
    alone.close()
    batch.close()

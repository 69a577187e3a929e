"""The geometry kernel's two forms (groups of few columns whose lanes share the
queries' edges, for batches that leave the chip idle; full groups with a thread
per query) give the same bits: an instance alone and the same instance in a
batch large enough for full groups, translating, static and rotating bodies."""
import numpy as np
import pytest

from paper_1711_11361_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("case", ["cylinder", "triangle", "piston", "naca", "channel"])
def test_alone_equals_in_a_large_batch(case):
    from paper_1711_11361_gb300 import mb
    if case == "naca":
        prob, fill = inputs.c3_naca(120), inputs.small_case("piston", 128)
    elif case == "channel":
        prob, fill = inputs.c1_advection(90), inputs.c1_advection(128)
    else:
        prob, fill = inputs.small_case(case, 101), inputs.small_case("piston", 128)
    alone, batch = mb.Sim(prob, mb.FP64), mb.Sim([prob] + [fill] * 60, mb.FP64)   # 60 x 128 / 8 columns: over 6 x 152
    for _ in range(3):
        alone.step()
        batch.step()
    a, b = alone.read_state(0, alpha=True), batch.read_state(0, alpha=True)
    assert np.array_equal(a["Q"], b["Q"], equal_nan=True) and np.array_equal(a["alpha"], b["alpha"])
    ra, rb = (np.sort(s.band_records(0), order="cell") for s in (alone, batch))
    for f in ("cell", "flags", "aA", "aB", "aM", "bown", "d", "nx", "ny", "wx", "wy"):
        assert np.array_equal(ra[f], rb[f]), f
    alone.close()
    batch.close()

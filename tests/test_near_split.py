"""The split of a line into the cells whose update reads body data and the
others (csrc/mb3_near.h), enumerated on the CPU: every line length up to 40,
body region and kind of side, one-cell periodic lines included."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1711_11361_gb300", "csrc")
SOURCE = """
#include "mb3_near.h"
extern "C" int faults(int nal, int r0, int rn, int periodic) {
    const mb3::Near N = mb3::near_span(r0, rn, nal, periodic != 0);
    int bad = 0, count = 0;
    for (int m = 0; m < nal; ++m) {
        // by the definition: within two cells before the region to two after its last face
        bool want = false;
        for (int q = r0 - 2; rn > 0 && q < r0 + rn + 3; ++q) want = want || (periodic ? ((q % nal) + nal) % nal == m : q == m);
        const bool got = mb3::near_pos(N, m, nal);
        bad += got != want;
        count += got;
        // the cells that the second pass takes: each of them once
        int times = 0;
        for (int q = N.a; q < N.a + N.len; ++q) times += (periodic ? ((q % nal) + nal) % nal : q) == m;
        bad += times != (want ? 1 : 0);
    }
    return bad + (count != N.len);
}
"""


@pytest.fixture(scope="module")
def faults(tmp_path_factory):
    d = tmp_path_factory.mktemp("near")
    src, lib = d / "near.cpp", d / "near.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-std=c++17", "-I", CSRC, "-o", str(lib), str(src)])
    return ctypes.CDLL(str(lib)).faults


@pytest.mark.parametrize("periodic", [0, 1])
def test_every_cell_is_updated_by_one_pass(faults, periodic):
    for nal in range(1, 41):
        for r0 in range(nal):
            for rn in range(0, nal - r0 + 1):
                assert faults(nal, r0, rn, periodic) == 0, (nal, r0, rn)

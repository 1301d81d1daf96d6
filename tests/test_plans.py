"""Launch plans (csrc/fc_plan.h), compiled here with the host compiler and driven from Python: rings, tile arithmetic, key splits, routes."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2311_08263_b200 import build

WRAP = """
#include "fc_plan.h"
extern "C" {
unsigned int last_copy_parity(int issued, int stages, int stage) { return fc::last_copy_parity(issued, stages, stage); }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = os.path.join(d, "wrap.cpp"), os.path.join(d, "plan.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", build.CSRC, src, "-o", so])
    return C.CDLL(so)


@pytest.mark.parametrize("stages", [1, 2, 3, 4, 6])
def test_parity_that_a_wait_for_the_copies_in_flight_asks_for(plan, stages):
    """After n completed phases a wait for parity p passes if p is that of phase n - 1.  Of `issued` requests, all but the last into a
    stage have landed: the wait must not pass; with that one landed it must."""
    for issued in range(1, 4 * stages + 2):
        for stage in range(min(stages, issued)):
            phases = len(range(stage, issued, stages))
            p = plan.last_copy_parity(issued, stages, stage)
            assert (phases - 1 - 1) % 2 != p and (phases - 1) % 2 == p

"""Launch plans (csrc/fc_plan.h), compiled here with the host compiler and driven from Python: rings, tile arithmetic, key splits, routes."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2311_08263_b200 import build

WRAP = """
#include "fc_plan.h"
#include <chrono>
#include <thread>
extern "C" {
unsigned int last_copy_parity(int issued, int stages, int stage) { return fc::last_copy_parity(issued, stages, stage); }
int ranges_exact(int units, int clusters) { return fc::ranges_exact(units, clusters, 8); }
// Bounds of the column ranges that differ from exact division; the largest range in *most.
int wrong_bounds(int units, int clusters, int *most) {
  const int parts = fc::column_ranges(units, clusters, 8);
  const unsigned int inv = fc::reciprocal(parts);
  int wrong = 0;
  *most = 0;
  for (int t = 0; t < parts; ++t) {
    const int b = fc::quotient(t * units, inv), e = fc::quotient((t + 1) * units, inv);
    if (b != (int)((long long)t * units / parts) || e != (int)((long long)(t + 1) * units / parts)) ++wrong;
    if (e - b > *most) *most = e - b;
  }
  return wrong;
}
// Two threads raise a limit to `a` and, begun a little later but finished at once, to `b`; the limit that stands.
long long raised_by_two(long long a, long long b) {
  fc::RisingLimit limit;
  long long stands = 0;
  auto raise = [&](long long n, int ms) {
    limit.raise(3, (size_t)n, [&](size_t v) { std::this_thread::sleep_for(std::chrono::milliseconds(ms)); stands = (long long)v; return 0; });
  };
  std::thread t(raise, a, 60);
  std::this_thread::sleep_for(std::chrono::milliseconds(20));
  raise(b, 0);
  t.join();
  return stands;
}
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = os.path.join(d, "wrap.cpp"), os.path.join(d, "plan.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-shared", "-fPIC", "-I", build.CSRC, src, "-o", so])
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


@pytest.mark.parametrize("a,b", [(100, 200), (200, 100)])
def test_limit_raised_by_two_threads_is_the_higher_one(plan, a, b):
    """Shared-memory limits of a kernel: contexts on different threads, windows of different length."""
    plan.raised_by_two.restype = C.c_longlong
    assert plan.raised_by_two(C.c_longlong(a), C.c_longlong(b)) == 200


@pytest.mark.parametrize("clusters", [16, 33, 37])
def test_column_ranges_by_reciprocals_are_exact_where_they_are_used(plan, clusters):
    """Every number of units that is let through has exact bounds and tiles of at most eight units; 125,000 (a vocabulary of two
    million) has neither and is not."""
    most = C.c_int(0)
    for units in list(range(1, 3000, 7)) + list(range(3000, 200000, 1013)):
        if plan.ranges_exact(units, clusters):
            assert plan.wrong_bounds(units, clusters, C.byref(most)) == 0
            assert most.value <= 8 * clusters
    assert plan.wrong_bounds(125000, 33, C.byref(most)) > 0 and not plan.ranges_exact(125000, 33)
    assert plan.ranges_exact(16032, clusters) and plan.ranges_exact(1792, clusters)

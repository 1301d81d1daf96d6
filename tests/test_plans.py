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
// fit: [2][9], clusters of 0 .. 8 CTAs with two CTAs per SM, then with one; returns splits, negative with half the ring
int short_plan(int tiles, int units, int head_dim, const int *fit) {
  int splits;
  bool deep;
  fc::short_plan(tiles, units, head_dim, 4, 148, [&](int s, bool d) { return (long long)fit[(d ? 9 : 0) + s]; }, splits, deep);
  return deep ? splits : -splits;
}
int one_writer_pays(int d, int qd, int kvd, int f, int rows, int cached, int fused) {
  const int shape[7][2] = {{qd, d}, {kvd, d}, {kvd, d}, {d, qd}, {f, d}, {f, d}, {d, f}};
  return fc::one_writer_pays(fc::stage_fill(shape, 7, 33), 2ll * d * (2ll * qd + 2ll * kvd + 3ll * f), rows, cached, fused != 0);
}
int stream_splits(int tiles, int units, int spare, const int *fit) {
  return fc::stream_splits(tiles, units, spare != 0, [&](int s) { return fit[s]; });
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


# what cudaOccupancyMaxActiveClusters says on a B200 (with two CTAs per SM less a sixteenth)
FIT = (C.c_int * 18)(0, 296, 138, 87, 66, 52, 42, 34, 30, 0, 148, 74, 45, 33, 26, 22, 15, 15)


@pytest.mark.parametrize("head_dim", [64, 128])
def test_key_splits_all_run_at_once(plan, head_dim):
    """Whatever the units and tiles: no more clusters than run at the same time, no CTA without a tile for its warps, never more than
    eight splits; and units of at most an SM each keep the whole ring unless a warp has more than two tiles."""
    for units in range(1, 400):
        for tiles in list(range(0, 70)) + [94, 250, 1000]:
            got = plan.short_plan(tiles, units, head_dim, FIT)
            s = abs(got)
            assert 1 <= s <= 8 and (s == 1 or s <= (tiles + 3) // 4)
            if s > 1:
                assert units <= FIT[(9 if got > 0 else 0) + s]
            if got > 0:
                assert units * s <= 148
            elif units <= 148:
                assert tiles > 8


@pytest.mark.parametrize("head_dim,units,tiles,want", [
    (128, 32, 25, 4), (128, 32, 250, 4), (128, 40, 250, 3), (128, 64, 25, -4), (128, 80, 125, -3), (128, 96, 63, 1), (128, 128, 64, 1), (128, 160, 90, -1),
    (64, 32, 20, 4), (64, 32, 94, -7), (64, 64, 32, -4), (64, 128, 64, -2),
    (64, 20, 32, 6), (64, 24, 32, 5), (64, 28, 32, 4), (64, 36, 22, 3), (64, 36, 57, -6), (128, 16, 47, 6), (128, 24, 25, 5), (128, 48, 47, -5), (128, 48, 10, 2),
])
def test_key_splits_of_the_measured_shapes(plan, head_dim, units, tiles, want):
    assert plan.short_plan(tiles, units, head_dim, FIT) == want


@pytest.mark.parametrize("shape,few,mid,many", [
    # d, heads x head_dim, kv heads x head_dim, d_ffn: rows up to 8, 9 to 16, 33 to 64 through one writer (17 to 32 always)
    ((2048, 2048, 256, 5632), 1, 1, 1),
    ((4096, 4096, 4096, 11008), 1, 1, 1),
    ((5120, 5120, 5120, 13824), 0, 1, 0),
    ((4352, 4352, 256, 8192), 0, 0, 0),            # a little over 33 x 8 units of 16 rows: two column ranges, stages half full
    ((4608, 4608, 512, 9216), 0, 0, 0),
    ((4352, 4352, 4352, 9600), 0, 0, 0),
    ((4608, 4608, 4608, 12288), 0, 0, 0),
    ((4864, 4864, 4864, 12928), 0, 1, 0),
    ((4224, 4224, 4224, 11264), 1, 1, 1),
    ((4096, 4096, 1024, 22016), 1, 1, 1),
    ((6656, 6656, 6656, 17920), 1, 1, 0),
    ((8192, 8192, 1024, 28672), 1, 1, 0),
    ((1024, 1024, 256, 2816), 1, 1, 1),
    ((3072, 3072, 1024, 8192), 1, 1, 1),
])
def test_route_of_the_measured_shapes(plan, shape, few, mid, many):
    for rows, want in ((1, few), (8, few), (9, mid), (16, mid), (17, 1), (32, 1), (33, many), (64, many)):
        assert plan.one_writer_pays(*shape, rows, 100, 1) == want, rows
        assert plan.one_writer_pays(*shape, rows, 8000, 0) == want, rows


def test_streaming_splits_leave_a_spare_only_where_it_is_asked_for(plan):
    """Two CTAs per SM, a sixteenth left out.  Behind the dense GEMMs 66 units take four splits and 136 two, which just fit; behind a
    persistent launch they take fewer or more, whatever leaves a thirty-second free.  Elsewhere the spare changes nothing."""
    for units, tiles, splits in ((66, 127, 4), (136, 126, 2), (42, 63, 6), (52, 63, 5), (34, 126, 7)):
        assert plan.stream_splits(tiles, units, 0, FIT) == splits
        with_spare = plan.stream_splits(tiles, units, 1, FIT)
        assert with_spare != splits and (units + units // 32 <= FIT[with_spare] or units > FIT[with_spare] or with_spare == 1)
    for units in (32, 40, 64, 80, 96, 128, 160, 320):
        for tiles in (1, 2, 8, 26, 63, 126, 250):
            assert plan.stream_splits(tiles, units, 0, FIT) == plan.stream_splits(tiles, units, 1, FIT)


@pytest.mark.parametrize("shape,rows,crossing", [
    # cached keys where the two routes cost the same (measured between 1000, 3000, 5000 and 8000)
    ((4352, 4352, 4352, 9600), 1, 4300), ((4352, 4352, 4352, 9600), 8, 2800), ((4352, 4352, 4352, 9600), 16, 2000),
    ((4352, 4352, 4352, 11520), 1, 4000), ((4352, 4352, 4352, 11520), 8, 2400), ((4608, 4608, 4608, 12288), 1, 2600),
    ((5120, 5120, 5120, 13824), 1, 2000), ((5120, 5120, 5120, 13824), 8, 600),
])
def test_long_caches_in_front_of_the_fused_attention_change_the_route(plan, shape, rows, crossing):
    assert plan.one_writer_pays(*shape, rows, crossing + 800, 1) == 1
    assert plan.one_writer_pays(*shape, rows, max(crossing - 800, 0), 1) == 0
    assert plan.one_writer_pays(*shape, rows, 8000, 0) == 0

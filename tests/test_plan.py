"""The host-side splits of a step (csrc/plan.h), compiled on their own."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRAP = """
#include "plan.h"
extern "C" int grid(long long N, int sms, int waits) { return ktune::shared_grid(N, sms, waits != 0); }
extern "C" int small_step(long long N, int D) { return ktune::small_step(N, D); }
extern "C" void bins(const long long *units, int n, int bins, long long chunk, long long piece, long long *out,
                     int *first, int *counts) {
  std::vector<ktune::Cut> c;
  std::vector<int> f;
  ktune::cut_bins(std::vector<int64_t>(units, units + n), bins, chunk, piece, &c, &f);
  counts[0] = (int)c.size();
  counts[1] = (int)f.size();
  for (size_t i = 0; i < c.size(); ++i) {
    out[3 * i] = c[i].search;
    out[3 * i + 1] = c[i].lo;
    out[3 * i + 2] = c[i].hi;
  }
  for (size_t i = 0; i < f.size(); ++i) first[i] = f[i];
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = d / "plan.cc", d / "plan.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2102_05297_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    return C.CDLL(str(lib))


@pytest.mark.parametrize("sms", [1, 3, 132, 152])
@pytest.mark.parametrize("waits", [0, 1])
def test_grids_leave_room_for_other_searches(plan, sms, waits):
    """Every grid fits the GPU and takes no more than one chunk of 4,096 per CTA where
    the GPU has the SMs; small spaces leave most of the GPU free."""
    for N in [1, 2, 4097, 5120, 16384, 16385, 40960, 77824, 77825, 155648, 155649, 162816, 204288, 245760, 262143]:
        g = plan.grid(N, sms, waits)
        assert 1 <= g <= sms
        assert -(-N // g) <= 4096 or g >= sms - 4
        if sms == 152:
            assert g <= max(16, -(-N // 1024))
            assert g <= 148                # a step may start while others draw
            if not waits:
                assert g <= max(38, -(-N // 4096))


def cut(plan, units, bins, chunk, piece):
    n = 4096
    out = (C.c_longlong * (3 * n))()
    first = (C.c_int * n)()
    counts = (C.c_int * 2)()
    plan.bins((C.c_longlong * len(units))(*units), len(units), bins, C.c_longlong(chunk), C.c_longlong(piece), out,
              first, counts)
    items = [(out[3 * i], out[3 * i + 1], out[3 * i + 2]) for i in range(counts[0])]
    return items, list(first[:counts[1]])


def cost(items, chunk, piece):
    return sum(piece + -(-(hi - lo) // chunk) * chunk for _, lo, hi in items)


@pytest.mark.parametrize("units,bins,chunk,piece", [
    ([500] * 64, 152, 4096, 1024), ([1000] * 40, 152, 4096, 1024), ([6], 152, 4096, 1024), ([0, 0], 152, 4096, 1024),
    ([40960, 500] * 32, 152, 4096, 1024), ([40960] * 16, 152, 2048, 1024), ([0, 3600, 0, 196608], 608, 3072, 1024),
    ([196608, 3600, 500, 16384] * 8, 152, 4096, 1024), ([3600] * 64, 10, 4096, 1024), ([74] * 32, 152, 1, 1),
    ([27648, 3, 1] * 21, 152, 1, 1)])
def test_bins_of_a_batch(plan, units, bins, chunk, piece):
    """Every search whole and in order; no bin more than a chunk and a search's staging
    above an even share; no search shares a bin while there are bins for each."""
    items, first = cut(plan, units, bins, chunk, piece)
    at = {i: 0 for i in range(len(units))}
    order = [i for i, _, _ in items]
    assert order == sorted(order)
    for i, lo, hi in items:
        assert lo == at[i] < hi
        at[i] = hi
    assert [at[i] for i in range(len(units))] == units
    assert first[0] == 0 and first[-1] == len(items) and len(first) - 1 <= bins
    loads = [cost(items[a:b], chunk, piece) for a, b in zip(first, first[1:])]
    assert all(x > 0 for x in loads)
    if not items:
        return
    even = sum(loads) / bins
    assert max(loads) <= max(chunk + piece, even + chunk + 2 * piece)
    if sum(-(-u // chunk) for u in units) <= bins:
        assert max(loads) == chunk + piece


def test_one_cta_only_where_trees_come_in_few_groups(plan):
    for D in range(0, 13):
        assert [plan.small_step(n, D) for n in (1, 2048, 2049, 4096, 4097)] == [1, 1, 1, 1, 0]
    assert [plan.small_step(n, 13) for n in (1, 2048, 2049, 4096)] == [1, 1, 0, 0]
    assert not any(plan.small_step(n, 14) for n in (1, 1024, 2048, 4096))

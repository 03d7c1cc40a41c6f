"""Rules that size a launch, compiled from the engine's header for the host."""

import ctypes
import os
import subprocess

import pytest

from conftest import ROOT
from paper_2602_20748_gb300 import build

MAX_BLOCKS = 608


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text("""#include "rpq_internal.h"
extern "C" int grid(int nw, unsigned groups, unsigned n, unsigned long long edges) {
  return rpq::bfs_grid(608, nw, groups, n, edges);
}
extern "C" int staged(int nw, unsigned groups, unsigned states, int by_source) {
  return rpq::lanes_staged(nw, groups, states, by_source != 0);
}
// Labels 0 and 1 with `longer` and `shorter` chunked rows each and `light` edges
// in the others, a launch that takes label 0: 1 its longer rows are chunked, 2 its
// shorter ones too, 4 its rows are walked.
extern "C" int chunked(unsigned n, unsigned longer, unsigned shorter, unsigned light, unsigned groups,
                       unsigned long long starts, int there, int lanes_staged) {
  static unsigned rec;
  rpq::ChunkLists c;
  c.rec = &rec;
  c.shorter = there ? 2 * shorter : 0;
  const unsigned listed = there ? shorter : 0;
  c.off = {0, longer, longer + listed, 2 * longer + listed, 2 * longer + 2 * listed};
  c.light = {light, 100 * n};
  c.shorter_rows = {shorter, shorter};
  rpq::BfsParams p{};
  p.n = n;
  p.L = 2;
  p.G = groups;
  p.q.n_states = 1;
  p.q.in_begin[1] = 1;
  p.q.in_label[0] = 0;
  rpq::set_chunks(p, c, starts, lanes_staged != 0);
  const bool shorts = p.heavy_row == rpq::HEAVY_ROW, walk = p.walk_rows;
  if (p.hchunk != &rec || p.hchunk_beg[0] != 0 || p.hchunk_end[0] != longer + (shorts ? shorter : 0) ||
      p.hchunk_beg[1] != longer + listed || (!shorts && p.heavy_row != rpq::LONG_ROW))
    return -1;
  c.rec = nullptr;
  rpq::set_chunks(p, c, starts, lanes_staged != 0);
  if (p.hchunk || !p.walk_rows) return -2;
  return 1 | (shorts ? 2 : 0) | (walk ? 4 : 0);
}
""")
    cuda = os.path.join(os.path.dirname(os.path.realpath(build._nvcc())), "..", "include")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{build.CSRC}", f"-I{build.INCLUDE}", f"-I{cuda}",
                    str(d / "rules.cpp"), "-o", str(d / "rules.so")], check=True)
    lib = ctypes.CDLL(str(d / "rules.so"))
    lib.grid.argtypes = [ctypes.c_int, ctypes.c_uint, ctypes.c_uint, ctypes.c_ulonglong]
    lib.chunked.argtypes = [ctypes.c_uint] * 5 + [ctypes.c_ulonglong, ctypes.c_int, ctypes.c_int]
    return lib


@pytest.mark.parametrize("nw,groups", [(1, 1), (1, 16), (4, 1), (4, 4), (4, 16)])
@pytest.mark.parametrize("n", [1, 1000, 4096, 1 << 20])
def test_grid_grows_with_vertices_and_edges(rules, nw, groups, n):
    # 5 edges per vertex: one vertex per sub-warp, as without edges
    sparse = rules.grid(nw, groups, n, 5 * n)
    assert sparse == rules.grid(nw, groups, n, 0) and 1 <= sparse <= MAX_BLOCKS
    grids = [rules.grid(nw, groups, n, d * n) for d in (5, 16, 64, 256, 1000, 4000)]
    assert grids == sorted(grids) and grids[-1] <= MAX_BLOCKS
    # 4 million edges are spread over every block, whatever the number of vertices
    assert rules.grid(nw, groups, n, 4_000_000) == MAX_BLOCKS


def test_staged_lane_levels_need_a_full_row_of_lanes(rules):
    assert [rules.staged(4, g, 8, 1) for g in (1, 4, 8, 9, 16)] == [0, 0, 0, 1, 1]
    assert not any((rules.staged(1, 16, 8, 1), rules.staged(4, 16, 9, 1), rules.staged(4, 16, 8, 0)))


K, BIG = 1 << 15, 1 << 17


@pytest.mark.parametrize("n,longer,shorter,light,groups,starts,there,want", [
    (K, 3, 0, 0, 2, 100, 1, 1), (K, 3, 1, 0, 2, 100, 1, 3), (K, 3, K // 8, 0, 2, 100, 1, 3), (K, 3, K // 8 + 1, 0, 2, 100, 1, 5),
    (K, 0, K - 9, 0, 16, 4096, 1, 5), (K - 8, 3, K // 2, 0, 2, 100, 1, 3), (K - 8, 3, K // 2, 0, 1, 100, 1, 5),
    (K, 3, 50, 0, 1, 31, 1, 1), (K, 3, 50, 0, 1, 32, 1, 3), (K, 3, 50, 0, 2, 100, 0, 1), (K, 3, K, 0, 1, 1, 0, 5),
    (BIG, 3, 50, 8 * BIG, 2, 300, 1, 3), (BIG, 3, 50, 8 * BIG + 1, 2, 300, 1, 7),
    (BIG, 3, 50, 8 * BIG + 1, 4, 1000, 1, 7), (BIG, 3, 50, 16 * BIG, 5, 1200, 1, 3),
    (BIG, 3, 50, 16 * BIG + 1, 16, 4096, 1, 7), (BIG - 8, 3, 50, 20 * BIG, 2, 300, 1, 3)])
def test_rows_that_are_chunked_and_rows_that_are_walked(rules, n, longer, shorter, light, groups, starts, there, want):
    assert rules.chunked(n, longer, shorter, light, groups, starts, there, 0) == want


def test_staged_lane_levels_keep_the_chunks(rules):
    assert rules.chunked(K, 3, K, 0, 12, 3000, 1, 1) == 3

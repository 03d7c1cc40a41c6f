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
""")
    cuda = os.path.join(os.path.dirname(os.path.realpath(build._nvcc())), "..", "include")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{build.CSRC}", f"-I{build.INCLUDE}", f"-I{cuda}",
                    str(d / "rules.cpp"), "-o", str(d / "rules.so")], check=True)
    lib = ctypes.CDLL(str(d / "rules.so"))
    lib.grid.argtypes = [ctypes.c_int, ctypes.c_uint, ctypes.c_uint, ctypes.c_ulonglong]
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

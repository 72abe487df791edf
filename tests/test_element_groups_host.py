"""Host test of the element groups of the sliced H X (csrc/element_groups.h,
compiled here): every element in one group, the groups that the grids of the
workloads have, and a bounded search on dense patterns."""
import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_03416_gb300", "csrc")
SOURCE = r"""
#include "element_groups.h"
extern "C" int groups(int M, const int64_t* row_ptr, const int32_t* col, int G, int32_t* out) {
  const std::vector<int32_t> g = dg::group_elements(M, row_ptr, col, G);
  std::copy(g.begin(), g.end(), out);
  return (int)g.size();
}
"""


@pytest.fixture(scope="module")
def group(tmp_path_factory):
    d = tmp_path_factory.mktemp("groups")
    (d / "g.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "g.so"), str(d / "g.cpp")],
                   check=True)
    lib = ctypes.CDLL(str(d / "g.so"))

    def call(C, G):
        C = np.asarray(C, dtype=bool)
        row_ptr = np.concatenate([[0], np.cumsum(C.sum(1))]).astype(np.int64)
        col = np.nonzero(C)[1].astype(np.int32)
        out = np.empty(len(C) * G, dtype=np.int32)
        n = lib.groups(len(C), row_ptr.ctypes.data_as(ctypes.c_void_p), col.ctypes.data_as(ctypes.c_void_p), G,
                       out.ctypes.data_as(ctypes.c_void_p))
        g = out[:n].reshape(-1, G)
        assert np.array_equal(np.sort(g[g >= 0]), np.arange(len(C)))
        return g

    return call


def grid(gx, gy, gz, wrap):
    M = gx * gy * gz
    C = np.zeros((M, M), dtype=bool)
    at = lambda x, y, z: (x % gx) + gx * ((y % gy) + gy * (z % gz))  # noqa: E731
    for x in range(gx):
        for y in range(gy):
            for z in range(gz):
                for a in (-1, 0, 1):
                    for b in (-1, 0, 1):
                        for c in (-1, 0, 1):
                            if wrap or (0 <= x + a < gx and 0 <= y + b < gy and 0 <= z + c < gz):
                                C[at(x, y, z), at(x + a, y + b, z + c)] = True
    return C


def unions(C, g):
    return np.array([C[[k for k in row if k >= 0]].any(0).sum() for row in g])


def test_grid_groups(group):
    """8 x 8 x 8 elements with 27 neighbours: pairs have 36, fours 48 (2 x 2)."""
    C = grid(8, 8, 8, True)
    assert (unions(C, group(C, 2)) == 36).all() and (unions(C, group(C, 4)) == 48).all()


@pytest.mark.parametrize("G", [2, 4, 8])
@pytest.mark.parametrize("shape", [(1, 1, 1), (7, 1, 1), (5, 3, 1), (3, 3, 3)])
@pytest.mark.parametrize("wrap", [True, False])
def test_every_element_once(group, shape, wrap, G):
    group(grid(*shape, wrap), G)


@pytest.mark.parametrize("chance", [0.0, 0.01, 0.25, 1.0])
def test_dense_patterns_are_grouped_quickly(group, chance):
    """1400 elements. With every neighbour tried at every level this took seconds."""
    rng = np.random.default_rng(1)
    C = np.triu(rng.random((1400, 1400)) < chance, 1)
    C = C | C.T | np.eye(1400, dtype=bool)
    t = time.perf_counter()
    g = group(C, 8)
    assert time.perf_counter() - t < 1.0
    if chance == 1.0:
        assert (g >= 0).all()

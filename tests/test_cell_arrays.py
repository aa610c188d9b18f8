"""The host-built arrays of trees and Voronoi grids (csrc/rt_cells.h, compiled as
C++) keep every load of the walks in range: ropes name nodes, node words name
children, the sorted pass's order of the cells is a permutation and its points
lie in their cells."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1410_1629_gb300 import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_1629_gb300", "csrc")

SHIM = f'''
#include "{CSRC}/rt_cells.h"
#include <cstring>
using namespace rtk;
extern "C" int order(int kind, const void* data, long long n_nodes, long long n_cells, const double* bounds, int* rank, float* point, int* id) {{
  CellOrder o(n_cells);
  bool ok = true;
  std::vector<int32_t> rope;
  std::vector<float> box;
  if (kind == 0) ok = order_octree((const int32_t*)data, bounds, o);
  else if (kind == 1) ok = bintree_walk_arrays((const int32_t*)data, n_nodes, n_cells, bounds, rope, box, o);
  else order_voronoi((const float*)data, bounds, o);
  if (!ok) return 0;
  for (size_t i = 0; i < o.rank.size(); ++i) {{
    point[3 * i] = o.cell[i].x; point[3 * i + 1] = o.cell[i].y; point[3 * i + 2] = o.cell[i].z;
    id[i] = o.cell[i].id;
  }}
  std::memcpy(rank, o.rank.data(), o.rank.size() * sizeof(int));
  return (int)o.rank.size();
}}
extern "C" void walk_arrays(const int32_t* word, long long n_nodes, long long n_cells, const double* bounds, int32_t* rope,
                            float* box) {{
  std::vector<int32_t> r;
  std::vector<float> b;
  CellOrder o(n_cells);
  bintree_walk_arrays(word, n_nodes, n_cells, bounds, r, b, o);
  std::memcpy(rope, r.data(), r.size() * sizeof(int32_t));
  std::memcpy(box, b.data(), b.size() * sizeof(float));
}}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cells")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-fsanitize=undefined",
                    "-fno-sanitize-recover=all", str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


def _order(lib, kind, data, n_cells, bounds):
    rank, point, ident = np.full(n_cells, -7, np.int32), np.zeros((n_cells, 3), np.float32), np.zeros(n_cells, np.int32)
    b = np.ascontiguousarray(bounds, dtype=np.float64)
    n = lib.order(kind, data.ctypes.data_as(ctypes.c_void_p), ctypes.c_longlong(len(data)), ctypes.c_longlong(n_cells),
                  b.ctypes.data_as(ctypes.c_void_p),
                  *(a.ctypes.data_as(ctypes.c_void_p) for a in (rank, point, ident)))
    return n, rank, point, ident


def _bintree(which):
    if which == "clumpy":
        return W.clumpy_bintree(n_particles=2000, n_samples=60_000, target_leaves=3000, max_level=6, n_lambda=1).grid
    rng = np.random.default_rng(3)
    bounds = [-1.3, 0.9, 0.1, 2.2, -3.0, 5.0]
    if which == "one leaf":
        return W.build_bintree(bounds, lambda lo, hi, d: np.zeros(len(lo), bool), lambda lo, hi: np.ones(len(lo)), 4)[0]
    return W.build_bintree(bounds, lambda lo, hi, d: rng.uniform(size=len(lo)) < 0.85, lambda lo, hi: np.ones(len(lo)), 14,
                           axis_of=lambda lo, hi, d: rng.integers(0, 3, len(lo)))[0]


def _octree(which):
    if which == "clumpy":
        return W.clumpy_octree(n_particles=2000, n_samples=60_000, target_leaves=3000, max_level=6, n_lambda=1).grid
    rng = np.random.default_rng(4)
    keep = 0.0 if which == "one leaf" else 0.5
    return W.build_octree([-1.3, 0.9, 0.1, 2.2, -3.0, 5.0], lambda lo, hi, l: rng.uniform(size=len(lo)) < max(keep, (l == 0) * keep * 2),
                          lambda lo, hi: np.ones(len(lo)), 7)[0]


def _permutation(n, rank, ident, n_cells):
    assert n == n_cells
    assert np.array_equal(np.sort(ident), np.arange(n_cells))
    assert np.array_equal(rank[ident], np.arange(n_cells))


def _descend(grid, point):
    """The leaf that holds a point (FP32 halving, ties to the upper child)."""
    lo, hi = np.float32(grid.bounds[0::2]).copy(), np.float32(grid.bounds[1::2]).copy()
    node = 0
    while grid.child[node] >= 0:
        axes = [int(grid.split_axis[node])] if grid.kind == "bintree" else [0, 1, 2]
        oct_ = 0
        for k, a in enumerate(axes):
            mid = np.float32(0.5) * (lo[a] + hi[a])
            if point[a] >= mid:
                oct_ |= 1 << k
                lo[a] = mid
            else:
                hi[a] = mid
        node = grid.child[node] + oct_
    assert np.all(lo < point) and np.all(point < hi)
    return -grid.child[node] - 1


@pytest.mark.parametrize("which", ["clumpy", "random axes", "one leaf"])
def test_bintree_arrays(lib, which):
    g = _bintree(which)
    n_nodes, n = len(g.child), g.n_cells
    inner = g.child >= 0
    word = np.where(inner, g.child.astype(np.int64) * 4 + np.where(inner, g.split_axis, 0), g.child).astype(np.int32)
    assert np.all(word[inner] >= 0) and np.array_equal(word[inner] >> 2, g.child[inner])  # the shift keeps its bits
    assert np.all((word[inner] & 3) <= 2) and np.all((word[inner] >> 2) + 1 < n_nodes)
    assert np.all(-word[~inner].astype(np.int64) - 1 < n)
    rope, box = np.full((n, 6), -7, np.int32), np.full((n_nodes, 2, 4), np.nan, np.float32)
    b = np.ascontiguousarray(g.bounds, dtype=np.float64)
    lib.walk_arrays(word.ctypes.data_as(ctypes.c_void_p), ctypes.c_longlong(n_nodes), ctypes.c_longlong(n),
                    b.ctypes.data_as(ctypes.c_void_p), rope.ctypes.data_as(ctypes.c_void_p), box.ctypes.data_as(ctypes.c_void_p))
    assert np.all((rope >= -1) & (rope < n_nodes))
    lo, hi = box[:, 0, :3], box[:, 1, :3]
    assert np.all(lo < hi)  # every node has its box
    leaf_node = np.empty(n, np.int64)
    leaf_node[-g.child[~inner] - 1] = np.flatnonzero(~inner)
    for a in range(3):
        others = [c for c in range(3) if c != a]
        for up in range(2):
            r = rope[:, 2 * a + up]
            face = (hi if up else lo)[leaf_node, a]
            edge = np.float32(g.bounds[2 * a + up])
            assert np.array_equal(r < 0, face == edge)  # no rope exactly at the domain's boundary
            m = r >= 0
            assert np.array_equal((lo if up else hi)[r[m], a], face[m])  # the node begins at the face
            for c in others:  # and covers it
                assert np.all(lo[r[m], c] <= lo[leaf_node[m], c]) and np.all(hi[leaf_node[m], c] <= hi[r[m], c])
    k, rank, point, ident = _order(lib, 1, word, n, g.bounds)
    _permutation(k, rank, ident, n)
    for i in range(0, n, max(1, n // 300)):
        assert _descend(g, point[i]) == ident[i]


@pytest.mark.parametrize("which", ["clumpy", "random", "one leaf"])
def test_octree_order(lib, which):
    g = _octree(which)
    child = np.ascontiguousarray(g.child, dtype=np.int32)
    k, rank, point, ident = _order(lib, 0, child, g.n_cells, g.bounds)
    _permutation(k, rank, ident, g.n_cells)
    for i in range(0, g.n_cells, max(1, g.n_cells // 300)):
        assert _descend(g, point[i]) == ident[i]


@pytest.mark.parametrize("kind", [0, 1])
def test_a_leaf_met_twice_gives_no_order(lib, kind):
    """Two parents that name the same children: no order (the walks then start in
    place); leaves that no parent names come last."""
    kids = 2 if kind else 8
    scale = 4 if kind else 1
    child = np.full(1 + 2 * kids, 0, np.int32)
    child[0] = 1 * scale
    child[1] = child[2] = (1 + kids) * scale
    child[3:] = -1 - np.arange(len(child) - 3)
    n, *_ = _order(lib, kind, child, len(child) - 3, [0, 1] * 3)
    assert n == 0
    child[2] = -1 - (len(child) - 3)
    n, rank, _, ident = _order(lib, kind, child, len(child) - 2, [0, 1] * 3)
    _permutation(n, rank, ident, len(child) - 2)
    child = np.concatenate([child, [-1 - (len(child) - 2)]]).astype(np.int32)  # named by no parent
    n, rank, _, ident = _order(lib, kind, child, len(child) - 2, [0, 1] * 3)
    _permutation(n, rank, ident, len(child) - 2)
    assert ident[-1] == len(child) - 3


@pytest.mark.parametrize("n_sites", [1, 2, 700])
def test_voronoi_order(lib, n_sites):
    rng = np.random.default_rng(n_sites)
    site = np.zeros((n_sites, 4), np.float32)
    site[:, :3] = rng.uniform(-1.0, 1.0, (n_sites, 3))
    site[0, :3] = 1.0  # on the domain's upper corner
    n, rank, point, ident = _order(lib, 2, site, n_sites, [-1, 1] * 3)
    _permutation(n, rank, ident, n_sites)
    assert np.array_equal(point, site[ident, :3])

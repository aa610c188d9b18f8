// Host-built arrays of the grids that are no box of planes (octrees, k-d trees,
// Voronoi grids): the order of the cells that the sorted peel-off pass starts
// its walks in, and the ropes and node boxes of the k-d tree walk.  Plain C++
// (tests compile it without CUDA).
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <memory>
#include <utility>
#include <vector>

namespace rtk {

// A point strictly inside a cell and the cell's id (the device reads it as
// float4 with the id's bits in w).
struct CellPoint {
  float x, y, z;
  int32_t id;
};

// An order of the cells that keeps neighbouring cells together: the place of
// every cell, and per place its cell.
struct CellOrder {
  std::vector<int> rank;
  std::unique_ptr<CellPoint[]> cell;

  explicit CellOrder(long long n_cells) : rank((size_t)n_cells, -1), cell(new CellPoint[(size_t)n_cells]) {}
};

// Fills an order, cell after cell (its own copies of the pointers and the count:
// the traversals below keep them in registers).
struct CellAppender {
  int* rank;
  CellPoint* cell;
  size_t n_cells;
  int n = 0;

  explicit CellAppender(CellOrder& o) : rank(o.rank.data()), cell(o.cell.get()), n_cells(o.rank.size()) {}
  // False if the cell has a place already (a node with two parents).
  bool append(long long id, float x, float y, float z) {
    if (rank[id] >= 0) return false;
    rank[id] = n;
    cell[n++] = CellPoint{x, y, z, (int32_t)id};
    return true;
  }
  // Cells of nodes that no parent names come last: no walk starts there.
  void append_rest(const double bounds[6]) {
    for (size_t i = 0; (size_t)n < n_cells && i < n_cells; ++i)
      if (rank[i] < 0) append((long long)i, (float)bounds[0], (float)bounds[2], (float)bounds[4]);
  }
};

// A tree's node and its box, with the device's FP32 halving.
struct TreeItem {
  long long node;
  float lo[3], hi[3];
};
inline TreeItem tree_root(const double bounds[6]) {
  TreeItem it;
  it.node = 0;
  for (int a = 0; a < 3; ++a) {
    it.lo[a] = (float)bounds[2 * a];
    it.hi[a] = (float)bounds[2 * a + 1];
  }
  return it;
}
inline bool append_leaf(CellAppender& order, int32_t word, const float (&lo)[3], const float (&hi)[3]) {
  return order.append(-(long long)word - 1, 0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2]));
}

// Octree leaves depth-first.  child[n] >= 0: the first of n's eight children,
// < 0: leaf -(child[n] + 1) (checked by the caller: in range, every child after
// its parent).  False if a leaf is met twice.
inline bool order_octree(const int32_t* child, const double bounds[6], CellOrder& out) {
  CellAppender order(out);
  // an inner node's leaves are placed from its own entry of the stack
  struct Inner {
    int32_t first;  // of its children
    int next;       // the child to visit
    float lo[3], mid[3], hi[3];
  };
  std::vector<Inner> stack;
  stack.reserve(32);
  const auto enter = [&](int32_t first, const float (&lo)[3], const float (&hi)[3]) {
    Inner it;
    it.first = first;
    it.next = 0;
    for (int a = 0; a < 3; ++a) {
      it.lo[a] = lo[a];
      it.hi[a] = hi[a];
      it.mid[a] = 0.5f * (lo[a] + hi[a]);
    }
    stack.push_back(it);
  };
  const TreeItem root = tree_root(bounds);
  if (child[0] < 0) append_leaf(order, child[0], root.lo, root.hi);
  else enter(child[0], root.lo, root.hi);
  while (!stack.empty()) {
    Inner& it = stack.back();
    if (it.next == 8) {
      stack.pop_back();
      continue;
    }
    const int o = it.next++;
    const int32_t v = child[(size_t)(it.first + o)];
    float lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
      lo[a] = (o >> a) & 1 ? it.mid[a] : it.lo[a];
      hi[a] = (o >> a) & 1 ? it.hi[a] : it.mid[a];
    }
    if (v >= 0) enter(v, lo, hi);
    else if (!append_leaf(order, v, lo, hi)) return false;
  }
  order.append_rest(bounds);
  return true;
}

// The two children of a k-d tree node (word: first child << 2 | split axis).
inline void split_node(const TreeItem& it, int32_t word, TreeItem& lower, TreeItem& upper) {
  const int a = word & 3;
  lower = upper = it;
  lower.node = word >> 2;
  upper.node = lower.node + 1;
  lower.hi[a] = upper.lo[a] = 0.5f * (it.lo[a] + it.hi[a]);
}

// Voronoi sites in Morton order, 10 bits per axis, sites of equal keys by
// index: a counting sort by ten key bits at a time.  site: x, y, z and one more
// float per site.
inline void order_voronoi(const float* site, const double bounds[6], CellOrder& out) {
  CellAppender order(out);
  const size_t n = out.rank.size();
  std::vector<std::pair<unsigned, int>> keys(n), sorted(n);
  for (size_t i = 0; i < n; ++i) {
    unsigned key = 0;
    for (int a = 0; a < 3; ++a) {
      const double u = (site[4 * i + (size_t)a] - bounds[2 * a]) / (bounds[2 * a + 1] - bounds[2 * a]);
      const unsigned v = (unsigned)std::min(1023.0, std::max(0.0, 1024.0 * u));
      for (int bit = 0; bit < 10; ++bit) key |= ((v >> bit) & 1u) << (3 * bit + a);
    }
    keys[i] = {key, (int)i};
  }
  for (int shift = 0; shift < 30; shift += 10) {
    std::vector<size_t> at(1025, 0);
    for (const auto& o : keys) ++at[((o.first >> shift) & 1023u) + 1];
    for (size_t k = 1; k < at.size(); ++k) at[k] += at[k - 1];
    for (const auto& o : keys) sorted[at[(o.first >> shift) & 1023u]++] = o;
    keys.swap(sorted);
  }
  for (const auto& o : keys) {
    const float* p = &site[4 * (size_t)o.second];
    order.append(o.second, p[0], p[1], p[2]);
  }
}

// Node boxes [n_nodes][2][4] (lo, 0, hi, 0) and the ropes of the k-d tree walk
// [n_cells][6]: per leaf and face (2 axis + upper) the node across it that
// covers it, the sibling of the ancestor whose split made the face, or -1 at the
// domain's boundary.  Going down, the lower child's rope across its upper face
// on the split axis is the upper child and the other way round; the other faces
// inherit.  On the way the leaves' order, depth-first (the traversal waits on
// the node words: a second one for the order would take as long); false, and no
// order, if a leaf is met twice.
inline bool bintree_walk_arrays(const int32_t* word, long long n_nodes, long long n_cells, const double bounds[6],
                                std::vector<int32_t>& rope, std::vector<float>& box, CellOrder& out) {
  CellAppender order(out);
  struct Item {
    TreeItem t;
    int32_t r[6];
  };
  rope.assign((size_t)n_cells * 6, -1);
  box.assign((size_t)n_nodes * 8, 0.0f);
  Item root;
  root.t = tree_root(bounds);
  for (int f = 0; f < 6; ++f) root.r[f] = -1;
  std::vector<Item> stack(1, root);
  bool whole = true;
  while (!stack.empty()) {
    const Item it = stack.back();
    stack.pop_back();
    for (int a = 0; a < 3; ++a) {
      box[8 * (size_t)it.t.node + (size_t)a] = it.t.lo[a];
      box[8 * (size_t)it.t.node + 4 + (size_t)a] = it.t.hi[a];
    }
    const int32_t v = word[(size_t)it.t.node];
    if (v < 0) {
      for (int f = 0; f < 6; ++f) rope[(size_t)(-(long long)v - 1) * 6 + (size_t)f] = it.r[f];
      whole = append_leaf(order, v, it.t.lo, it.t.hi) && whole;
      continue;
    }
    Item lower = it, upper = it;
    split_node(it.t, v, lower.t, upper.t);
    lower.r[2 * (v & 3) + 1] = (int32_t)upper.t.node;
    upper.r[2 * (v & 3)] = (int32_t)lower.t.node;
    stack.push_back(lower);
    stack.push_back(upper);
  }
  if (whole) order.append_rest(bounds);
  return whole;
}

}  // namespace rtk

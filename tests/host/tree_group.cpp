// Host harness for tests/test_tree_group_host.py: the group query of the tree neighbour list
// (csrc/tree_rows.cuh: the box of a group of particles against node boxes, up to 32 nodes
// of one level from the top of a stack at a time) restated for one thread over the boxes
// and distances of csrc/tree_core.cuh, which the kernels use.
#include <cstdint>
#include <vector>

#include "../../paper_1308_5587_gb300/csrc/tree_core.cuh"

using namespace gbmd;

extern "C" uint32_t box_gap(uint32_t a, uint32_t b, uint32_t lo, uint32_t hi) {
  return tree_box_gap(a, b, lo, hi);
}

namespace {
int level(int node) { return 31 - __builtin_clz((unsigned)node); }
}

// Leaves within sqrt(r2) of the box of members first .. first + count - 1 (of `order`), in
// the order of the visits; returns their number, -1 when the bound on the rounds ran out.
// *deepest: the most entries of the stack.
extern "C" int group_leaves(int n, const uint32_t* u, const int* order, const double* L, float r2,
                            int first, int count, int* leaves, int* deepest) {
  const int P = tree_leaves(n);
  std::vector<TreeBox> box(2 * (size_t)P);
  for (int b = 0; b < P; ++b) {
    TreeBox t = tree_empty_box();
    for (int m = b * TREE_LEAF; m < n && m < (b + 1) * TREE_LEAF; ++m)
      tree_box_add(t, u[3 * order[m]], u[3 * order[m] + 1], u[3 * order[m] + 2]);
    box[P + b] = t;
  }
  for (int k = P - 1; k >= 1; --k) box[k] = tree_box_union(box[2 * k], box[2 * k + 1]);
  TreeBox me = tree_empty_box();
  for (int m = first; m < first + count; ++m)
    tree_box_add(me, u[3 * order[m]], u[3 * order[m] + 1], u[3 * order[m] + 2]);
  float fs[3];
  for (int a = 0; a < 3; ++a) fs[a] = (float)(L[a] / 4294967296.0);
  std::vector<int> stack;
  const int start = P < 32 ? P : 32;   // the deepest level with at most 32 nodes
  for (int k = start - 1; k >= 0; --k) stack.push_back(start + k);
  int found = 0, left = 2 * P + 64;
  *deepest = (int)stack.size();
  while (!stack.empty()) {
    if (--left < 0) return -1;
    std::vector<int> run;   // one level, in order from the top
    while (run.size() < 32 && run.size() < stack.size()) {
      const int here = stack[stack.size() - 1 - run.size()];
      if (!run.empty() && level(here) != level(run[0])) break;
      run.push_back(here);
    }
    stack.resize(stack.size() - run.size());
    std::vector<int> in;
    for (int k : run) {
      const TreeBox& b = box[k];
      if (tree_box_empty(b)) continue;
      const float gx = (float)tree_box_gap(me.x, me.x2, b.x, b.x2) * fs[0];
      const float gy = (float)tree_box_gap(me.y, me.y2, b.y, b.y2) * fs[1];
      const float gz = (float)tree_box_gap(me.z, me.z2, b.z, b.z2) * fs[2];
      if (gx * gx + gy * gy + gz * gz < r2) in.push_back(k);
    }
    if (run[0] >= P) {
      for (int k : in) leaves[found++] = k - P;
    } else {
      for (size_t k = in.size(); k-- > 0;) {
        stack.push_back(2 * in[k] + 1);
        stack.push_back(2 * in[k]);
      }
    }
    if ((int)stack.size() > *deepest) *deepest = (int)stack.size();
  }
  return found;
}

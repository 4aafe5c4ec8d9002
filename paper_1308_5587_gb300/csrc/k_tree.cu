// k_tree.cu -- the tree neighbour list (Section 5: nlist.tree, a bounding volume
// hierarchy per particle type, for size-disperse systems).
//
// After the cell sort (k_bin .. k_cellsort, type-major bins, Morton order of the
// particles inside a bin), type t's particles are members[tree_first[t] ..
// + tree_n[t]) in Morton order of cells, then of particles.  Its tree is the
// implicit complete binary tree of tree_core.cuh over them, TREE_LEAF particles per
// leaf.  Two kernels, both no-ops for systems not rebuilding or on the cell list:
//   k_tree_build  one thread per leaf: the leaf's box and a copy of its particles
//                 (position, index) in leaf order, then up the tree: the second child
//                 to arrive at a node writes its box (an arrival counter per node,
//                 which that child resets); no thread waits for another;
//   k_tree_nlist  one warp per group of particles (tree_rows.cuh), the types with the
//                 longest queries first (they would otherwise finish last): for every
//                 type t, the leaves of t's tree within r_list(t_i, t) of the group, then
//                 the same pair decision as the cell list (nlist_core.cuh).  The row holds
//                 the neighbours in (type, cell order) order.
// A traversal examines each node at most once, so 2 P nodes bound it; passing the
// bound (which cannot happen) would stop it and set DEV_TREE.
#include "launch.cuh"
#include "tree_rows.cuh"

namespace gbmd {

KernelCall make_call(void* f, int grid, int block, size_t smem);

template <typename T>
static void put(KernelCall& k, const T& v) {
  static_assert(sizeof(T) <= 16, "arg too large");
  memcpy(k.store[k.nargs], &v, sizeof(T));
  ++k.nargs;
}

__global__ void __launch_bounds__(TILE_P) k_tree_build(const SysDev* __restrict__ sysv,
                                                       const Tile* __restrict__ tiles,
                                                       GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  count(s, t, ctl);
  if (!rebuilding(s) || !s.tree || (int)threadIdx.x >= t.count) return;
  tree_leaf(s, q_at(s, step_of(s.flags)), t.first + threadIdx.x);
}

// tiles: `count` groups of one type from group `first` on; pad = type, + 256 where a
// group is a single particle
__global__ void __launch_bounds__(TREE_WARPS * 32) k_tree_nlist(const SysDev* __restrict__ sysv,
                                                                const Tile* __restrict__ tiles,
                                                                GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  count(s, t, ctl);
  __shared__ TreeWarp sm[TREE_WARPS];
  __shared__ TreeTable tab;
  if (!block_rebuilding(s) || !s.tree) return;
  tree_table(s, tab);
  __syncthreads();
  const int w = threadIdx.x >> 5;
  if (w >= t.count) return;
  const int ty = t.pad & 255, per = t.pad & 256 ? 1 : TREE_G, first = (t.first + w) * per;
  unsigned long long nb = 0;
  const int over = tree_rows(s, ty, first, min(per, s.tree_n[ty] - first), per, sm[w], tab, nb);
  if (over > 0) {
    atomicMax(&s.flags->overflow_need, over);
    atomicCAS(&s.flags->error, 0, (int)DEV_OVERFLOW);
  }
  if (over < 0) atomicCAS(&s.flags->error, 0, (int)DEV_TREE);
  for (int o = 16; o > 0; o >>= 1) nb += __shfl_down_sync(0xffffffffu, nb, o);
  if ((threadIdx.x & 31) == 0 && nb) atomicAdd(&s.flags->nb_total, nb);
}

KernelCall tree_build_call(const SysDev* d, const Tile* tiles_l, int ntiles, GroupCtl* ctl) {
  KernelCall k = make_call((void*)k_tree_build, ntiles, TILE_P, 0);
  put(k, d); put(k, tiles_l); put(k, ctl);
  return k;
}

KernelCall tree_nlist_call(const SysDev* d, const Tile* tiles_g, int ntiles, GroupCtl* ctl) {
  KernelCall k = make_call((void*)k_tree_nlist, ntiles, TREE_WARPS * 32, 0);
  put(k, d); put(k, tiles_g); put(k, ctl);
  return k;
}

}  // namespace gbmd

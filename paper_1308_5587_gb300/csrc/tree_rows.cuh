// tree_rows.cuh -- the device pieces of the tree neighbour list: a leaf's box and climb,
// and the rows of a group of particles by one warp.  Shared by the kernels of k_tree.cu
// and the cooperative rebuild (k_lists.cu).
#pragma once
#include "launch.cuh"
#include "nlist_core.cuh"

namespace gbmd {

// fixed-point coordinate on [0, 2^32): the box [-L/2, L/2) in order
__device__ __forceinline__ uint32_t tree_u(int q) { return (uint32_t)q ^ 0x80000000u; }

// a node box, perhaps written by another thread of this launch: from L2, past L1
__device__ __forceinline__ TreeBox load_box_l2(const TreeBox* p) {
  const uint4 a = __ldcg(reinterpret_cast<const uint4*>(p));
  const uint4 b = __ldcg(reinterpret_cast<const uint4*>(p) + 1);
  TreeBox r;
  r.x = a.x; r.y = a.y; r.z = a.z; r.pad0 = 0u;
  r.x2 = b.x; r.y2 = b.y; r.z2 = b.z; r.pad1 = 0u;
  return r;
}

// leaf g (numbered over all types of the system): its box, the copy of its particles,
// and the boxes above it whose other child has arrived
__device__ __forceinline__ void tree_leaf(const SysDev& s, const int4* qv, int g) {
  int ty = 0;
  while (ty + 1 < s.ntypes && g >= s.tree_leaf0[ty + 1]) ++ty;
  const int P = s.tree_P[ty], b = g - s.tree_leaf0[ty];
  TreeBox* boxes = s.tree_box + s.tree_node0[ty];
  unsigned* arrive = s.tree_arrive + s.tree_node0[ty];
  const int first = s.tree_first[ty], nty = s.tree_n[ty];
  TreeBox box = tree_empty_box();
#pragma unroll
  for (int k = 0; k < TREE_LEAF; ++k) {
    const int m = b * TREE_LEAF + k;
    if (m < nty) {
      const int j = s.members[first + m];
      const int4 q = qv[j];
      tree_box_add(box, tree_u(q.x), tree_u(q.y), tree_u(q.z));
      s.tree_q[first + m] = make_int4(q.x, q.y, q.z, j);   // the leaf's own copy
    }
  }
  int node = P + b;
  boxes[node] = box;
  while (node > 1) {   // at most log2(P) levels
    __threadfence();   // this thread's box before its arrival
    const int parent = node >> 1;
    if (atomicAdd(&arrive[parent], 1u) == 0u) return;   // the sibling goes on
    arrive[parent] = 0u;   // both children are in: ready for the next build
    __threadfence();
    box = tree_box_union(load_box_l2(boxes + 2 * parent), load_box_l2(boxes + 2 * parent + 1));
    boxes[parent] = box;
    node = parent;
  }
}

// ---- rows: one warp per group of particles ----
// The query of one particle by one thread walks ~180 nodes (a large particle of a 1:10
// mixture a few thousand) in a dependent chain, 12 of 32 lanes active on average.  Here
// a warp queries for TREE_G consecutive particles of a type at once (neighbours in the
// sort order; one particle where a type is sparse beside its r_list, tree_single), a lane per node: the stack's top nodes of one level are tested together
// against the box of the group, and the children of those within reach go back on top.
// Popping only one level at a time keeps the leaves in ascending order, so a row holds
// its neighbours in (type, cell order) order as the thread's walk did.  Each particle's
// lanes then test the leaves' particles from a ring of 32.
// WCA 1:10, N = 100,100: a build 1,405 us with a walk per thread, 243 this way (ncu; 587
// before groups that span much of the box query one by one).
constexpr int TREE_STACK = 1088;   // 32 entries a level stay (at most 30 levels), 64 on top

struct TreeWarp {
  int stack[TREE_STACK];
  int leaf[64];      // leaves within reach, not tested yet
  int4 cand[32];     // their particles: x, y, z, j
};
// r_list^2 (1 -+ band) and r_list^2 per type pair
struct TreeTable {
  float lo[MAXT2], hi[MAXT2];
  double rl2[MAXT2];
};
// every thread of the block calls it; followed by a __syncthreads
__device__ __forceinline__ void tree_table(const SysDev& s, TreeTable& t) {
  if ((int)threadIdx.x < s.ntypes * s.ntypes) {
    const float rl2 = s.pf[threadIdx.x].rl2;
    t.lo[threadIdx.x] = rl2 * (1.0f - NL_BAND);
    t.hi[threadIdx.x] = rl2 * (1.0f + NL_BAND);
    t.rl2[threadIdx.x] = s.pd[threadIdx.x].rl2;
  }
}

// The rows of members first .. first + count - 1 (count <= per) of type ty, per = TREE_G
// or 1 particles at a time.  Returns the longest row past the capacity (0: none; -1: the
// traversal ran past its bound).  Every lane of the warp calls it.
__device__ __forceinline__ int tree_query_rows(const SysDev& s, int ty, int first, int count,
                                               int per, TreeWarp& sm, const TreeTable& tab,
                                               unsigned long long& nb) {
  const int lane = threadIdx.x & 31;
  // lanes of a particle: 32 / per; this lane's particle p and place c among its lanes
  const int lanes = 32 / per, shift = per == 1 ? 5 : 2;
  const int p = lane >> shift, c = lane & (lanes - 1);
  const bool valid = p < count;
  const int4 qi = s.tree_q[s.tree_first[ty] + first + (valid ? p : 0)];
  const int i = qi.w;
  const uint32_t ux = tree_u(qi.x), uy = tree_u(qi.y), uz = tree_u(qi.z);
  const uint32_t x0 = __reduce_min_sync(0xffffffffu, ux), x1 = __reduce_max_sync(0xffffffffu, ux);
  const uint32_t y0 = __reduce_min_sync(0xffffffffu, uy), y1 = __reduce_max_sync(0xffffffffu, uy);
  const uint32_t z0 = __reduce_min_sync(0xffffffffu, uz), z1 = __reduce_max_sync(0xffffffffu, uz);
  const float fs0 = s.fscale[0], fs1 = s.fscale[1], fs2 = s.fscale[2];
  const int cap = s.cap;
  const size_t group = (size_t)s.nl_stride * 4;
  int* const row = s.nl + (size_t)i * 4;
  int cnt = 0, bad = 0;
  for (int tj = 0; tj < s.ntypes; ++tj) {
    const int pr = ty * s.ntypes + tj;
    const float lo = tab.lo[pr], hi = tab.hi[pr];
    const int P = s.tree_P[tj], nty = s.tree_n[tj];
    const int4* leaves = s.tree_q + s.tree_first[tj];
    const TreeBox* boxes = s.tree_box + s.tree_node0[tj];
    int nleaf = 0;   // leaves waiting in sm.leaf (fewer than 8 between rounds)
    // the waiting leaves' particles, eight leaves at a time
    auto test = [&](int at, int m) {   // leaves sm.leaf[at .. at + m), m <= 8
      const int k = lane >> 2;   // TREE_LEAF = 4 lanes a leaf
      int4 q = make_int4(0, 0, 0, -1);
      if (k < m) {
        const int e = sm.leaf[at + k] * TREE_LEAF + (lane & 3);
        if (e < nty) q = leaves[e];
      }
      unsigned mine = 0u;   // this lane's hits: candidate e at bit 31 - e
      auto hit = [&](const int4& qj) -> bool {
        const float dx = (float)min_image_fixed(qi.x, qj.x) * fs0;
        const float dy = (float)min_image_fixed(qi.y, qj.y) * fs1;
        const float dz = (float)min_image_fixed(qi.z, qj.z) * fs2;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        return valid && qj.w >= 0 && qj.w != i && r2 < hi &&
               (r2 < lo || exact_within(s, i, qj.w, tab.rl2[pr]));
      };
      unsigned all;
      if (per == 1) {
        mine = hit(q) ? 0x80000000u >> lane : 0u;
        all = __reduce_or_sync(0xffffffffu, mine);
      } else {
        __syncwarp();   // the previous candidates have been read
        sm.cand[lane] = q;
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 8; ++e) {   // candidates c, c + 4, ..: one 64-byte read a turn
          const int at4 = 4 * e + c;
          if (hit(sm.cand[at4])) mine |= 0x80000000u >> at4;
        }
        all = mine | __shfl_xor_sync(0xffffffffu, mine, 1);
        all |= __shfl_xor_sync(0xffffffffu, all, 2);
      }
      while (mine) {
        const int e = __clz(mine);
        mine &= ~(0x80000000u >> e);
        const int at2 = cnt + (e ? __popc(all >> (32 - e)) : 0);
        const int j = per == 1 ? q.w : sm.cand[e].w;
        if (at2 < cap) row[(size_t)(at2 >> 2) * group + (at2 & 3)] = j;
      }
      cnt += __popc(all);
    };
    // the deepest level with at most 32 nodes, in order from the top of the stack
    const int start = P < 32 ? P : 32;
    __syncwarp();
    if (lane < start) sm.stack[start - 1 - lane] = start + lane;
    int top = start, left = 2 * P + 64;
    __syncwarp();
    while (top > 0) {
      if (--left < 0) { bad = 1; break; }
      const int here = lane < top ? sm.stack[top - 1 - lane] : 0;
      const int head = __shfl_sync(0xffffffffu, here, 0);
      const bool same = lane < top && __clz(here) == __clz(head);   // one level
      const unsigned run = __ballot_sync(0xffffffffu, same);
      const int m = run == 0xffffffffu ? 32 : __ffs(~run) - 1;
      bool in = false;
      if (lane < m) {
        const TreeBox b = load_box_l2(boxes + here);
        if (!tree_box_empty(b)) {
          const float gx = (float)tree_box_gap(x0, x1, b.x, b.x2) * fs0;
          const float gy = (float)tree_box_gap(y0, y1, b.y, b.y2) * fs1;
          const float gz = (float)tree_box_gap(z0, z1, b.z, b.z2) * fs2;
          in = gx * gx + gy * gy + gz * gz < hi;
        }
      }
      const unsigned ok = __ballot_sync(0xffffffffu, in);
      const int before = __popc(ok & ((1u << lane) - 1u)), total = __popc(ok);
      top -= m;
      __syncwarp();   // the popped entries have been read
      if (head >= P) {   // leaves, in ascending order
        if (in) sm.leaf[nleaf + before] = here - P;
        nleaf += total;
        __syncwarp();
        int at = 0;
        for (; nleaf - at >= 8; at += 8) test(at, 8);
        const int keep = nleaf - at;   // fewer than 8: to the front
        const int v = lane < keep ? sm.leaf[at + lane] : 0;
        __syncwarp();
        if (lane < keep) sm.leaf[lane] = v;
        nleaf = keep;
      } else {
        if (in) {
          const int e = top + 2 * (total - 1 - before);
          sm.stack[e + 1] = 2 * here;
          sm.stack[e] = 2 * here + 1;
        }
        top += 2 * total;
      }
      __syncwarp();
    }
    if (nleaf > 0) test(0, nleaf);
    __syncwarp();
  }
  int over = 0;
  if (valid && c == 0) {
    s.nn[i] = cnt < cap ? cnt : cap;
    s.q_build[i] = make_int4(qi.x, qi.y, qi.z, ty);
    nb += (unsigned long long)cnt;
    if (cnt > cap) over = cnt;
  }
  return bad ? -1 : over;   // `bad` is the same in every lane
}

// The same for a group of up to TREE_G particles.  Where the sort order jumps, a group
// can span much of the box, and its query would then visit every leaf in between (one
// such warp outlives the rest of the build): while the space within reach of its box is
// more than TREE_SPREAD times one particle's, the first half of it queries alone.  (Most
// groups hold one jump; querying their particles one by one took eight queries for the
// two to four of the halves: 40 steps with readouts, WCA 1:10, N = 100,100, 1,826 ->
// 1,580 us)
constexpr float TREE_SPREAD = 16.0f;
__device__ __forceinline__ int tree_rows(const SysDev& s, int ty, int first, int count, int per,
                                         TreeWarp& sm, const TreeTable& tab,
                                         unsigned long long& nb) {
  const int lane = threadIdx.x & 31;
  float hi = 3e38f;
  for (int t = 0; t < s.ntypes; ++t) hi = fminf(hi, tab.hi[ty * s.ntypes + t]);
  const float d = 2.0f * sqrtf(hi);
  auto spread = [&](int k, int m) -> bool {
    const int4 q = s.tree_q[s.tree_first[ty] + first + k + (lane < m ? lane : 0)];
    auto extent = [](int v, float fs) {
      const uint32_t u = tree_u(v);
      return (float)(__reduce_max_sync(0xffffffffu, u) - __reduce_min_sync(0xffffffffu, u)) * fs;
    };
    const float ex = extent(q.x, s.fscale[0]), ey = extent(q.y, s.fscale[1]), ez = extent(q.z, s.fscale[2]);
    return (ex + d) * (ey + d) * (ez + d) > TREE_SPREAD * d * d * d;
  };
  int over = 0;
  for (int k = 0; k < count;) {
    int m = count - k;
    while (m > 1 && spread(k, m)) m = (m + 1) / 2;
    const int r = tree_query_rows(s, ty, first + k, m, m == 1 ? 1 : per, sm, tab, nb);
    if (r < 0) return -1;
    over = max(over, r);
    k += m;
  }
  return over;
}

}  // namespace gbmd

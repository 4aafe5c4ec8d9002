// team_core.cuh -- teams of resident thread blocks: the barrier with its vote, and the
// list rebuild of one system by a team.
//
// A team is
//   * a thread-block cluster (hardware barrier, votes through distributed shared
//     memory): one per system, so a launch steps any number of systems side by side; or
//   * the whole grid of a cooperative launch (one system), for systems with more work
//     than one cluster's SMs should carry: arrivals on one counter, the last one
//     publishes the outcome.  Waits are bounded; one that runs out sets DEV_TEAM.
#pragma once
#include <cooperative_groups.h>

#include "nlist_split.cuh"
#include "nlist_warp.cuh"
#include "sort_core.cuh"
#include "step_core.cuh"
#include "tree_rows.cuh"

namespace gbmd {

constexpr int TEAM_SPIN = 1 << 22;   // polls of ~0.5 us: two seconds
enum : unsigned { VOTE_NEED = 1u, VOTE_BAD = 2u, VOTE_LOST = 4u };

// shared memory of the phases (one at a time; dynamic: more than 48 KB)
template <int T, int SLOTS>
union TeamSmem {
  SplitCell split[T / NS_T];
  WarpRing<false, SLOTS> warp[T / 32];
  struct { TreeWarp warp[T / 32]; TreeTable tab; } tree;
  int scan[32];
  double slots[NH_SLOTS];
  int queue[16 * T];   // FP64 force phase (k_force.cuh)
};

struct Team {
  int rank, size, cluster;   // this block, blocks, 0: the whole grid
  GroupCtl* ctl;
  unsigned gen;              // grid: generation last seen released
  int par;                   // cluster: which vote slots are in use
  unsigned* slot;            // [2][TEAM_MAX_CLUSTER] in shared memory
  unsigned* word;            // one word in shared memory

  // Every thread of every block of the team: all of them have arrived, what they wrote
  // is visible, and the votes are ORed (VOTE_LOST: a wait ran out; the team stops).
  __device__ __forceinline__ unsigned vote(unsigned mine) {
    unsigned v = 0u;
    if (__syncthreads_or((int)mine))   // mostly nobody votes: one barrier of the block
      v = (__syncthreads_or((int)(mine & VOTE_NEED)) ? VOTE_NEED : 0u) |
          (__syncthreads_or((int)(mine & VOTE_BAD)) ? VOTE_BAD : 0u);
    if (size == 1) return v;
    if (cluster) {
      namespace cg = cooperative_groups;
      cg::cluster_group cl = cg::this_cluster();
      unsigned* const my = slot + par * TEAM_MAX_CLUSTER;
      if ((int)threadIdx.x < size) cl.map_shared_rank(my, threadIdx.x)[rank] = v;
      cl.sync();
      for (int k = 0; k < size; ++k) v |= my[k];
      par ^= 1;   // the next vote writes the other slots: these may still be read
      return v;
    }
    if (threadIdx.x == 0) {
      // arrivals in the low 32 bits; the blocks that vote NEED and BAD above them
      const unsigned long long add = 1ull | ((unsigned long long)(v & VOTE_NEED) << 32) |
                                     ((unsigned long long)((v & VOTE_BAD) >> 1) << 48);
      unsigned long long all;
      asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], %2;"
                   : "=l"(all) : "l"(&ctl->team_arrive), "l"(add) : "memory");
      all += add;
      unsigned out;
      if ((unsigned)all == (unsigned)size) {
        out = (((all >> 32) & 0xffffu) ? VOTE_NEED : 0u) | ((all >> 48) ? VOTE_BAD : 0u);
        ctl->team_arrive = 0ull;
        const unsigned long long rel = ((unsigned long long)(gen + 1u) << 8) | out;
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&ctl->team_release), "l"(rel) : "memory");
      } else {
        out = VOTE_LOST;
        for (int k = 0; k < TEAM_SPIN; ++k) {
          unsigned long long rel;
          asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(rel) : "l"(&ctl->team_release) : "memory");
          if ((unsigned)(rel >> 8) == gen + 1u) {
            out = (unsigned)rel & 0xffu;
            break;
          }
        }
      }
      *word = out;
    }
    ++gen;
    __syncthreads();
    return *word;   // not written again before the next vote's first barrier
  }
};

// Exclusive scan of the bin counts by one block (PER bins a thread and turn)
template <int T>
__device__ __forceinline__ void scan_bins(const SysDev& s, int* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nc = s.nbins;
  int carry = 0;
  if (threadIdx.x == 0) {
    s.flags->nb_total = 0;
    s.flags->max_window = 0;
  }
  constexpr int PER = 4;
  for (int base = 0; base < nc; base += PER * T) {
    const int c = base + PER * (int)threadIdx.x;
    int v[PER], sum = 0;
#pragma unroll
    for (int k = 0; k < PER; k += 4) {
      if (c + k + 3 < nc) {
        const int4 q = *reinterpret_cast<const int4*>(s.cell_cnt + c + k);
        v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w;
      } else {
        for (int u = 0; u < 4; ++u) v[k + u] = c + k + u < nc ? s.cell_cnt[c + k + u] : 0;
      }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) sum += v[k];
    int x = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    __syncthreads();   // the previous turn's totals have been read
    if (lane == 31) sh[w] = x;
    __syncthreads();
    int before = carry;
    for (int k = 0; k < T / 32; ++k) {
      if (k < w) before += sh[k];
      carry += sh[k];
    }
    int e = before + x - sum;
#pragma unroll
    for (int k = 0; k < PER; ++k)
      if (c + k < nc) {
        s.cell_start[c + k] = e;
        s.cell_cursor[c + k] = e;
        s.cell_cnt[c + k] = 0;   // the next build
        e += v[k];
      }
  }
  if (threadIdx.x == 0) {
    s.cell_start[nc] = carry;
    s.cell_cursor[nc] = 0;   // the list build's work counter
  }
}

// The list rebuild (and re-sort) of the team's system at the positions of `step`;
// returns the last vote (BAD: a row passed the capacity, the flags say so).
template <int T, bool MULTI, int SLOTS>
__device__ __noinline__ unsigned team_rebuild(const SysDev& s, Team& tm, TeamSmem<T, SLOTS>& sm,
                                              SplitTable& tab, long long step, bool sort) {
  const int n = s.n;
  const int t0 = tm.rank * T + threadIdx.x, nt = tm.size * T;
  const int w0 = tm.rank * (T / 32) + (threadIdx.x >> 5), nw = tm.size * (T / 32);
  const int4* qv = q_at(s, step);
  for (int i = t0; i < n; i += nt) bin_one(s, qv, i);
  if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
  if (tm.rank == 0) scan_bins<T>(s, sm.scan);
  if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
  for (int i = t0; i < n; i += nt) scatter_one(s, i);
  if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
  for (int r = w0; r < s.nbins; r += nw) cellsort_one(s, qv, r);
  if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
  if (sort) {
    for (int k = t0; k < n; k += nt) permute_one(s, qv, k);
    if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
    for (int k = t0; k < n; k += nt) copyback_one(s, step, k);
    if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
  }
  unsigned long long nb = 0;
  int over = 0;
  int* const next = s.cell_cursor + s.nbins;   // work counter, set to 0 by the scan
  const int lane = threadIdx.x & 31;
  if (s.tree) {
    for (int g = t0; g < s.tree_leaves_total; g += nt) tree_leaf(s, qv, g);
    if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
    tree_table(s, sm.tree.tab);
    __syncthreads();
    for (int k = w0;;) {   // query groups, the types with the longest queries first
      int q = 0;
      if (lane == 0) q = nw + atomicAdd(next, 1);   // in flight during the query
      int at = k, o = 0, ty = 0, per = 1, groups = 0;
      for (; o < s.ntypes; ++o, at -= groups) {
        ty = s.tree_qtype[o];
        per = s.tree_single[ty] ? 1 : TREE_G;
        groups = (s.tree_n[ty] + per - 1) / per;
        if (at < groups) break;
      }
      if (o == s.ntypes) break;
      const int r = tree_rows(s, ty, at * per, min(per, s.tree_n[ty] - at * per), per,
                              sm.tree.warp[threadIdx.x >> 5], sm.tree.tab, nb);
      if (r < 0) atomicCAS(&s.flags->error, 0, (int)DEV_TREE);
      over = max(over, r);
      k = __shfl_sync(0xffffffffu, q, 0);
    }
  } else {
    // Four warps a cell (nlist_split) while that keeps every group of four warps to one
    // item; with more cells the team is busy anyway and a warp a cell needs fewer
    // instructions (N = 20,011 on the whole grid, 729 cells: 37 us by four warps in two
    // turns, 35 by one)
    const int g = threadIdx.x / NS_T, groups = tm.size * (T / NS_T);
    const int split = max(1, (n / s.ncells + 31) / 32);   // parts of a cell, 32 particles each
    if ((long long)s.nbins * split <= groups) {
      for (int k = tm.rank + g * tm.size; k < s.nbins * split; k += groups)
        over = max(over, nlist_split<MULTI>(s, k / split, k % split, split, g, sm.split[g], tab, nb));
    } else {
      // cells of uneven cost: after its first, a warp takes the next free cell
      for (int r = w0; r < s.nbins;) {
        int q = 0;
        if (lane == 0) q = nw + atomicAdd(next, 1);   // in flight during the build
        over = max(over, nlist_cell<MULTI, false, false>(s, r, sm.warp[threadIdx.x >> 5], nb));
        r = __shfl_sync(0xffffffffu, q, 0);
      }
    }
  }
  if (over > 0) {
    atomicMax(&s.flags->overflow_need, over);
    atomicCAS(&s.flags->error, 0, (int)DEV_OVERFLOW);
  }
  for (int o = 16; o > 0; o >>= 1) nb += __shfl_down_sync(0xffffffffu, nb, o);
  if ((threadIdx.x & 31) == 0 && nb) atomicAdd(&s.flags->nb_total, nb);
  return tm.vote(over > 0 ? VOTE_BAD : 0u);
}

}  // namespace gbmd

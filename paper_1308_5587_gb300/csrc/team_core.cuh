// team_core.cuh -- teams of resident thread blocks: the barrier with its vote, and the
// list rebuild of one system by a team.
//
// A team is
//   * a thread-block cluster (hardware barrier, votes through distributed shared
//     memory): one per system, so a launch steps any number of systems side by side; or
//   * the whole grid of a cooperative launch (one system), for systems with more work
//     than one cluster's SMs should carry, or a share of that grid (a batch whose
//     clusters would not all run at once): arrivals on one counter, the last one
//     publishes the outcome.  Waits are bounded; one that runs out sets DEV_TEAM.
#pragma once
#include <cooperative_groups.h>

#include "nlist_split.cuh"
#include "nlist_warp.cuh"
#include "sort_core.cuh"
#include "step_core.cuh"
#include "tree_rows.cuh"

namespace gbmd {

enum : unsigned { VOTE_NEED = 1u, VOTE_BAD = 2u, VOTE_LOST = 4u };
// polls of a wait between blocks through memory, ~0.5 us each: two seconds; then the wait
// is given up, the kernel returns and the system stops with DEV_TEAM
constexpr int TEAM_POLLS = 1 << 22;

// The team's cell sort takes buckets: the histogram's atomic places each particle in its
// bin's bucket, every block scans the counts for itself, and each bin is sorted out of
// its bucket into its final place: one barrier where count, scan and scatter take three.
// For up to SCAN_MAX bins with a mean of at most two thirds of a bucket; a bucket that
// runs over sends the rebuild to the separate phases.  The buckets lie in the re-sort's
// scratch.  With the even spread of the cells over the blocks (below), 50 steps with
// readouts: N = 64,000 1,872 -> 1,789 us; one list build of N = 20,011 with its
// readouts 464 -> 443.
constexpr int SCAN_MAX = 12288, BUCKET = 64;

// shared memory of the phases (one at a time; dynamic: more than 48 KB)
template <int T, int SLOTS>
union TeamSmem {
  SplitCell split[T / NS_T];
  WarpRing<false, SLOTS> warp[T / 32];
  struct { TreeWarp warp[T / 32]; TreeTable tab; } tree;
  struct { int start[SCAN_MAX + 1], warp[32]; } scan;
  double sums[NH_SUMS];
  int queue[16 * T];   // FP64 force phase (k_force.cuh)
};

struct Team {
  int rank, size, cluster;   // this block, blocks, 0: no cluster
  TeamSync* sync;
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
                   : "=l"(all) : "l"(&sync->arrive), "l"(add) : "memory");
      all += add;
      unsigned out;
      if ((unsigned)all == (unsigned)size) {
        out = (((all >> 32) & 0xffffu) ? VOTE_NEED : 0u) | (((all & ~TEAM_CLOSED) >> 48) ? VOTE_BAD : 0u);
        sync->arrive = all & TEAM_CLOSED;
        const unsigned long long rel = ((unsigned long long)(gen + 1u) << 8) | out;
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&sync->release), "l"(rel) : "memory");
      } else {
        out = VOTE_LOST;
        for (int k = all & TEAM_CLOSED ? TEAM_POLLS : 0; k < TEAM_POLLS; ++k) {
          unsigned long long rel;
          asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(rel) : "l"(&sync->release) : "memory");
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

// The same by every block for itself, into shared memory: start[0 .. nbins]
template <int T>
__device__ __forceinline__ void scan_own(const SysDev& s, int* start, int* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nc = s.nbins;
  for (int c = threadIdx.x; c < nc; c += T) start[c] = __ldcg(s.cell_cnt + c);
  __syncthreads();
  const int per = ((nc + T - 1) / T) | 1;   // consecutive bins of a thread (odd: no bank twice)
  const int c0 = min(nc, (int)threadIdx.x * per), c1 = min(nc, c0 + per);
  int sum = 0;
  for (int c = c0; c < c1; ++c) sum += start[c];
  int x = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[w] = x;
  __syncthreads();
  int e = x - sum;
  for (int k = 0; k < w; ++k) e += sh[k];
  for (int c = c0; c < c1; ++c) {
    const int m = start[c];
    start[c] = e;
    e += m;
  }
  if (threadIdx.x == 0) start[nc] = s.n;
  __syncthreads();
}

// The list rebuild (and re-sort) of the team's system at the positions of `step`;
// returns the last vote (BAD: a row passed the capacity, the flags say so).
template <int T, bool MULTI, int SLOTS>
__device__ __noinline__ unsigned team_rebuild(const SysDev& s, Team& tm, TeamSmem<T, SLOTS>& sm,
                                              SplitTable& tab, long long step, bool sort) {
  const int n = s.n;
  const int t0 = tm.rank * T + threadIdx.x, nt = tm.size * T;
  const int w = threadIdx.x >> 5, nw = tm.size * (T / 32);
  const int4* qv = q_at(s, step);
  // this block's bins
  const int r0 = (int)((long long)s.nbins * tm.rank / tm.size);
  const int r1 = (int)((long long)s.nbins * (tm.rank + 1) / tm.size);
  int* const bucket = reinterpret_cast<int*>(s.x_alt);   // 6 n entries
  const int bcap = (int)min((long long)BUCKET, 6ll * n / s.nbins);
  bool full = s.nbins > SCAN_MAX || bcap < 16 || 3ll * n > 2ll * bcap * s.nbins;
  if (full) {
    for (int i = t0; i < n; i += nt) bin_one(s, qv, i);
  } else {
    for (int i = t0; i < n; i += nt) full |= !bin_bucket(s, qv, i, bucket, bcap);
  }
  const unsigned v = tm.vote(full ? VOTE_NEED : 0u);
  if (v & VOTE_LOST) return VOTE_LOST;
  const bool direct = !(v & VOTE_NEED);
  if (direct) {
    scan_own<T>(s, sm.scan.start, sm.scan.warp);
    const int* const start = sm.scan.start;
    for (int r = r0 + (int)threadIdx.x; r < r1; r += T) s.cell_start[r] = start[r];
    if (tm.rank == 0 && threadIdx.x == 0) {
      s.cell_start[s.nbins] = n;
      s.cell_cursor[s.nbins] = 0;   // the list build's work counter
      s.flags->nb_total = 0;
      s.flags->max_window = 0;
    }
    for (int r = r0 + w; r < r1; r += T / 32)
      cellsort_one(s, qv, bucket + (size_t)r * bcap, start[r], start[r + 1] - start[r]);
  } else {
    if (tm.rank == 0) scan_bins<T>(s, sm.scan.warp);
    if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
    for (int i = t0; i < n; i += nt) scatter_one(s, i);
    if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
    for (int r = r0 + w; r < r1; r += T / 32) {
      const int b = s.cell_start[r];
      cellsort_one(s, qv, s.members_tmp + b, b, s.cell_start[r + 1] - b);
    }
  }
  if (tm.vote(0u) & VOTE_LOST) return VOTE_LOST;
  if (direct)   // every block has scanned the counts: empty for the next build
    for (int r = r0 + (int)threadIdx.x; r < r1; r += T) s.cell_cnt[r] = 0;
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
    // query groups, the types with the longest queries first and spread over the blocks
    for (int k = w * tm.size + tm.rank;;) {
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
    } else if (s.nbins <= nw) {
      // a cell to a warp: every block gets its share of them (before, 729 cells of N =
      // 20,011 kept 46 of 152 blocks busy, 2,744 of N = 64,000 115)
      const int r = r0 + w;
      if (r < r1) over = nlist_cell<MULTI, false, false>(s, r, sm.warp[w], nb);
    } else {
      // cells of uneven cost: after its first, a warp takes the next free cell
      for (int r = tm.rank * (T / 32) + w; r < s.nbins;) {
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

// k_lists.cu -- cell list (integer binning + stable counting sort in Morton cell
// order), optional re-sort of the particle arrays, and the Verlet neighbour list.
//
// The paper names the structure (md.nlist.cell, Listing 1) and that HOOMD builds
// cell lists with atomic operations (Section 5); it gives no algorithm.  Here:
//   * a particle's cell comes from its 32-bit fixed-point coordinate, integer only:
//     c_a = floor((q_a + 2^31) * nc_a / 2^32), cell width L_a / nc_a >= r_list_max;
//   * cells are numbered by their rank in Morton (Z-order) of (cx, cy, cz);
//   * counting sort: atomic histogram -> exclusive scan -> atomic scatter, then
//     each cell's members are sorted by (the particle's own 30-bit Morton code,
//     index), so the result is the order (cell rank, fine Morton code, index)
//     whatever order the atomics ran in, and consecutive members of a cell are
//     spatial neighbours (a warp of the force kernel gathers from fewer lines:
//     2% off the step kernel at KA 10^6);
//   * neighbour list: full list (both i->j and j->i), one warp per cell whose lanes
//     are the cell's particles; every lane tests the same candidate j of the
//     neighbouring cells at a time (warp-uniform loop, broadcast loads).  Keep
//     j != i with r^2 < r_list,ij^2 (strict), r_list,ij = r_cut,ij + r_buff.  The
//     test runs in FP32 on the fixed-point difference; candidates within a relative
//     band of 1e-5 of r_list^2 are decided again in FP64 with the same operations
//     (and rounding) as the brute-force reference definition.  Hits are appended in
//     candidate order, so a row does not depend on how r^2 was rounded.
#include <algorithm>

#include "launch.cuh"
#include "nlist_core.cuh"
#include "team_core.cuh"

namespace gbmd {

KernelCall make_call(void* f, int grid, int block, size_t smem);

template <typename T>
static void put(KernelCall& k, const T& v) {
  static_assert(sizeof(T) <= 16, "arg too large");
  memcpy(k.store[k.nargs], &v, sizeof(T));
  ++k.nargs;
}

__device__ __forceinline__ bool sorting(const SysDev& s) {
  const FlagWords w = load_flag_words(s.flags);
  return w.do_rebuild != 0 && w.do_sort != 0;
}

// The per-particle rebuild kernels (bin, scatter, permute, copyback) walk the tile
// table with a grid of at most WALK_BLOCKS blocks.  Warp 0 reads, for up to 32 of the
// block's next tiles at once, whether their system does this work (and counts the
// launch at each system's first tile); the block then works on those tiles only.  In
// a batch where a few members rebuild, the others' tiles then cost one parallel read,
// not a block each.
constexpr int WALK_BLOCKS = 152 * 8;

template <typename Active, typename Work>
__device__ __forceinline__ void walk_tiles(const SysDev* __restrict__ sysv,
                                           const Tile* __restrict__ tiles, int ntiles,
                                           GroupCtl* ctl, Active active, Work work) {
  __shared__ int act[32];
  if (threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(&ctl->launches, 1ull);
  for (int b0 = blockIdx.x; b0 < ntiles; b0 += 32 * gridDim.x) {
    __syncthreads();   // the previous round's act[] has been read
    if (threadIdx.x < 32) {
      const int b = b0 + threadIdx.x * gridDim.x;
      int a = 0;
      if (b < ntiles) {
        const Tile t = tiles[b];
        const SysDev& s = sysv[t.sys];
        if (t.first == 0) atomicAdd(&s.flags->launches, 1ull);
        a = active(s) ? 1 : 0;
      }
      act[threadIdx.x] = a;
    }
    __syncthreads();
    for (int l = 0; l < 32; ++l) {
      const int b = b0 + l * gridDim.x;
      if (b >= ntiles) break;
      if (!act[l]) continue;
      const Tile t = tiles[b];
      if ((int)threadIdx.x < t.count) work(sysv[t.sys], t.first + (int)threadIdx.x);
    }
  }
}

__global__ void __launch_bounds__(TILE_P) k_bin(const SysDev* __restrict__ sysv,
                                                const Tile* __restrict__ tiles, int ntiles,
                                                GroupCtl* ctl) {
  walk_tiles(sysv, tiles, ntiles, ctl, [](const SysDev& s) { return rebuilding(s); },
             [](const SysDev& s, int i) { bin_one(s, q_at(s, step_of(s.flags)), i); });
}

// ---- exclusive scan of the bin counts (one block per system) ----
__global__ void __launch_bounds__(SCAN_THREADS) k_scan(const SysDev* __restrict__ sysv,
                                                       const Tile* __restrict__ tiles,
                                                       GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  count(s, t, ctl);
  if (!rebuilding(s)) return;
  __shared__ int warp_tot[32];
  __shared__ int carry;
  if (threadIdx.x == 0) {
    carry = 0;
    s.flags->nb_total = 0;
    s.flags->max_window = 0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nc = s.nbins;
  // four bins per thread (one 16-byte load where all four exist; the buffers come
  // from cudaMalloc, so 16-byte aligned)
  for (int base = 0; base < nc; base += 4 * SCAN_THREADS) {
    const int c = base + 4 * threadIdx.x;
    int v[4];
    if (c + 3 < nc) {
      const int4 q = *reinterpret_cast<const int4*>(s.cell_cnt + c);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
      for (int k = 0; k < 4; ++k) v[k] = c + k < nc ? s.cell_cnt[c + k] : 0;
    }
    const int v4 = v[0] + v[1] + v[2] + v[3];
    int x = v4;
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
      int w = warp_tot[lane];
      for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
      }
      warp_tot[lane] = w;   // inclusive over warps
    }
    __syncthreads();
    int e[4];
    e[0] = carry + (wid ? warp_tot[wid - 1] : 0) + x - v4;
    e[1] = e[0] + v[0];
    e[2] = e[1] + v[1];
    e[3] = e[2] + v[2];
    if (c + 3 < nc) {
      const int4 q = make_int4(e[0], e[1], e[2], e[3]);
      *reinterpret_cast<int4*>(s.cell_start + c) = q;
      *reinterpret_cast<int4*>(s.cell_cursor + c) = q;
      *reinterpret_cast<int4*>(s.cell_cnt + c) = make_int4(0, 0, 0, 0);   // next build
    } else {
      for (int k = 0; k < 4; ++k) {
        if (c + k < nc) {
          s.cell_start[c + k] = e[k];
          s.cell_cursor[c + k] = e[k];
          s.cell_cnt[c + k] = 0;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) carry += warp_tot[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) s.cell_start[nc] = carry;
}

__global__ void __launch_bounds__(TILE_P) k_scatter(const SysDev* __restrict__ sysv,
                                                    const Tile* __restrict__ tiles, int ntiles,
                                                    GroupCtl* ctl) {
  walk_tiles(sysv, tiles, ntiles, ctl, [](const SysDev& s) { return rebuilding(s); }, scatter_one);
}

// ---- sort each bin's members (warp per bin) ----
__global__ void __launch_bounds__(CELLS_PER_TILE * 32) k_cellsort(const SysDev* __restrict__ sysv,
                                                                  const Tile* __restrict__ tiles,
                                                                  GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  count(s, t, ctl);
  const int w = threadIdx.x >> 5;
  if (!block_rebuilding(s) || w >= t.count) return;
  const int b = s.cell_start[t.first + w];
  cellsort_one(s, q_at(s, step_of(s.flags)), s.members_tmp + b, b, s.cell_start[t.first + w + 1] - b);
}

// ---- re-sort: gather every per-particle array into cell order ----
// Both kernels run at every rebuild and do work only when the system re-sorts (the
// tile walker makes that cheap when it does not).
__global__ void __launch_bounds__(TILE_P) k_permute(const SysDev* __restrict__ sysv,
                                                    const Tile* __restrict__ tiles, int ntiles,
                                                    GroupCtl* ctl) {
  walk_tiles(sysv, tiles, ntiles, ctl, [](const SysDev& s) { return sorting(s); },
             [](const SysDev& s, int k) { permute_one(s, q_at(s, step_of(s.flags)), k); });
}

__global__ void __launch_bounds__(TILE_P) k_copyback(const SysDev* __restrict__ sysv,
                                                     const Tile* __restrict__ tiles, int ntiles,
                                                     GroupCtl* ctl) {
  walk_tiles(sysv, tiles, ntiles, ctl, [](const SysDev& s) { return sorting(s); },
             [](const SysDev& s, int k) { copyback_one(s, step_of(s.flags), k); });
}

// ---- staged force tiles: the window of every aligned 2x2x2 block of cells ----
// One warp per block.  The window is the 4x4x4 cells around the block (the union
// of its cells' 27-cell stencils; distinct because every axis has >= 4 cells),
// listed with x fastest; each window cell contributes its member range, placed at
// a running offset.  The block's own cells have 8 consecutive Morton codes, so
// their members form one contiguous range.
__global__ void __launch_bounds__(256) k_blocks(const SysDev* __restrict__ sysv,
                                                const Tile* __restrict__ tiles, GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  count(s, t, ctl);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (!rebuilding(s) || !s.staged || w >= t.count) return;
  const int b = t.first + w;
  const int nb0 = s.nb[0], nb1 = s.nb[1];
  const int bx = b % nb0, by = (b / nb0) % nb1, bz = b / (nb0 * nb1);
  const int nc0 = s.nc[0], nc1 = s.nc[1], nc2 = s.nc[2];
  int st[2], cn[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int wi = lane + 32 * h;
    const int cx = (2 * bx - 1 + (wi & 3) + nc0) % nc0;
    const int cy = (2 * by - 1 + ((wi >> 2) & 3) + nc1) % nc1;
    const int cz = (2 * bz - 1 + (wi >> 4) + nc2) % nc2;
    const int r = s.lin2rank[(cz * nc1 + cy) * nc0 + cx];
    st[h] = s.cell_start[r];
    cn[h] = s.cell_start[r + 1] - st[h];
  }
  int p0 = cn[0], p1 = cn[1];   // inclusive prefixes
  for (int o = 1; o < 32; o <<= 1) {
    const int y0 = __shfl_up_sync(0xffffffffu, p0, o);
    const int y1 = __shfl_up_sync(0xffffffffu, p1, o);
    if (lane >= o) {
      p0 += y0;
      p1 += y1;
    }
  }
  const int tot0 = __shfl_sync(0xffffffffu, p0, 31);
  const int wtot = tot0 + __shfl_sync(0xffffffffu, p1, 31);
  s.blk_win[(size_t)b * WIN_CELLS + lane] = make_int2(st[0], p0 - cn[0]);
  s.blk_win[(size_t)b * WIN_CELLS + 32 + lane] = make_int2(st[1], tot0 + p1 - cn[1]);
  // the block's own cells: lanes 0..7 take (ox, oy, oz)
  int rk = 0x7fffffff;
  bool exists = false;
  if (lane < 8) {
    const int cx = 2 * bx + (lane & 1), cy = 2 * by + ((lane >> 1) & 1), cz = 2 * bz + (lane >> 2);
    exists = cx < nc0 && cy < nc1 && cz < nc2;
    if (exists) rk = s.lin2rank[(cz * nc1 + cy) * nc0 + cx];
  }
  const int nown = __popc(__ballot_sync(0xffffffffu, exists));
  for (int o = 16; o > 0; o >>= 1) rk = min(rk, __shfl_xor_sync(0xffffffffu, rk, o));
  if (lane == 0) {
    const int first = s.cell_start[rk];
    s.blk_info[b] = make_int4(first, s.cell_start[rk + nown] - first, wtot, 0);
    atomicMax(&s.flags->max_window, wtot);
    if (wtot > s.window_cap) atomicCAS(&s.flags->error, 0, (int)DEV_WINDOW);
  }
}

// ---- neighbour list: one warp per cell (nlist_warp.cuh) ----
template <bool MULTI, bool REL, bool STAGED>
__global__ void __launch_bounds__(CELLS_PER_TILE * 32, 3) k_nlist(const SysDev* __restrict__ sysv,
                                                                  const Tile* __restrict__ tiles,
                                                                  GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  count(s, t, ctl);
  __shared__ WarpRing<STAGED> sm[CELLS_PER_TILE];
  const int w = threadIdx.x >> 5;
  if (!block_rebuilding(s) || s.tree || w >= t.count) return;
  unsigned long long nb_sum = 0;
  const int over = nlist_cell<MULTI, REL, STAGED>(s, t.first + w, sm[w], nb_sum);
  if (over > 0) {
    atomicMax(&s.flags->overflow_need, over);
    atomicCAS(&s.flags->error, 0, (int)DEV_OVERFLOW);
  }
  for (int o = 16; o > 0; o >>= 1) nb_sum += __shfl_down_sync(0xffffffffu, nb_sum, o);
  if ((threadIdx.x & 31) == 0 && nb_sum) atomicAdd(&s.flags->nb_total, nb_sum);
}

// The builder for systems with few cells (nlist_split.cuh): one block a tile, for cell
// rank `first`, part `count` of `pad` parts.
template <bool MULTI>
__global__ void __launch_bounds__(NS_T, 6) k_nlist_split(const SysDev* __restrict__ sysv,
                                                         const Tile* __restrict__ tiles,
                                                         GroupCtl* ctl) {
  const Tile t = tiles[blockIdx.x];
  const SysDev& s = sysv[t.sys];
  if (t.count == 0) count(s, t, ctl);
  __shared__ SplitCell sc;
  __shared__ SplitTable tab;
  if (!block_rebuilding(s) || s.tree) return;
  split_table(s, tab);
  __syncthreads();
  unsigned long long nb = 0;
  const int over = nlist_split<MULTI>(s, t.first, t.count, t.pad, 0, sc, tab, nb);
  if (over > 0) {
    atomicMax(&s.flags->overflow_need, over);
    atomicCAS(&s.flags->error, 0, (int)DEV_OVERFLOW);
  }
  for (int o = 16; o > 0; o >>= 1) nb += __shfl_down_sync(0xffffffffu, nb, o);
  if ((threadIdx.x & 31) == 0 && nb) atomicAdd(&s.flags->nb_total, nb);
}

// ---- the whole rebuild of one system by the grid of a cooperative launch ----
// Runs after every step and returns at once unless the step asked for a rebuild: ~2 us
// then, against ~13 us for a graph's conditional node (64k particles, mixed: 33.1 us a
// step with the node and seven kernels in its body, 28.2 us with this kernel).
template <bool MULTI>
__global__ void __launch_bounds__(REBUILD_T, 1) k_rebuild(const SysDev* __restrict__ sysv,
                                                            GroupCtl* ctl) {
  constexpr int T = REBUILD_T;
  using Smem = TeamSmem<T, NL_SLOTS>;
  static_assert(sizeof(Smem) <= REBUILD_SMEM, "shared memory");
  const SysDev& s = sysv[0];
  // nothing of this launch writes these words, so every block decides alike
  const FlagWords fw = load_flag_words(s.flags);
  if (!fw.do_rebuild) return;
  extern __shared__ __align__(16) unsigned char rebuild_smem[];
  Smem& sm = *reinterpret_cast<Smem*>(rebuild_smem);
  __shared__ SplitTable tab;
  __shared__ unsigned word;
  Team tm;
  tm.cluster = 0;
  tm.size = (int)gridDim.x;
  tm.rank = (int)blockIdx.x;
  tm.sync = &ctl->team;
  tm.gen = (unsigned)(*(const volatile unsigned long long*)&ctl->team.release >> 8);
  tm.par = 0;
  tm.slot = nullptr;
  tm.word = &word;
  split_table(s, tab);
  __syncthreads();
  const unsigned r = team_rebuild<T, MULTI>(s, tm, sm, tab, step_of(s.flags), fw.do_sort != 0);
  if (tm.rank == 0 && threadIdx.x == 0) {
    if (r & VOTE_LOST) atomicCAS(&s.flags->error, 0, (int)DEV_TEAM);
    atomicAdd(&s.flags->launches, 1ull);
    atomicAdd(&ctl->launches, 1ull);
  }
}

// ---- launch descriptors ----
#define SIMPLE_CALL(name, kern, block)                                           \
  KernelCall name(const SysDev* d, const Tile* tl, int ntiles, GroupCtl* ctl) { \
    KernelCall k = make_call((void*)kern, ntiles, block, 0);                    \
    put(k, d); put(k, tl); put(k, ctl);                                          \
    return k;                                                                    \
  }
SIMPLE_CALL(scan_call, k_scan, SCAN_THREADS)
SIMPLE_CALL(cellsort_call, k_cellsort, CELLS_PER_TILE * 32)
#define WALK_CALL(name, kern)                                                  \
  KernelCall name(const SysDev* d, const Tile* tl, int ntiles, GroupCtl* ctl) { \
    KernelCall k = make_call((void*)kern, std::min(ntiles, WALK_BLOCKS), TILE_P, 0);   \
    put(k, d); put(k, tl); put(k, ntiles); put(k, ctl);                            \
    return k;                                                                    \
  }
WALK_CALL(bin_call, k_bin)
WALK_CALL(scatter_call, k_scatter)
WALK_CALL(permute_call, k_permute)
WALK_CALL(copyback_call, k_copyback)
#undef WALK_CALL
SIMPLE_CALL(blocks_call, k_blocks, 256)
#undef SIMPLE_CALL

void* rebuild_func(bool multi) { return multi ? (void*)k_rebuild<true> : (void*)k_rebuild<false>; }
KernelCall rebuild_call(const SysDev* d, int blocks, GroupCtl* ctl, bool multi) {
  KernelCall k = make_call(rebuild_func(multi), blocks, REBUILD_T, REBUILD_SMEM);
  k.cooperative = true;
  put(k, d); put(k, ctl);
  return k;
}

KernelCall nlist_split_call(const SysDev* d, const Tile* tl, int ntiles, GroupCtl* ctl, bool multi) {
  KernelCall k = make_call(multi ? (void*)k_nlist_split<true> : (void*)k_nlist_split<false>, ntiles,
                           NS_T, 0);
  put(k, d); put(k, tl); put(k, ctl);
  return k;
}

KernelCall nlist_call(const SysDev* d, const Tile* tl, int ntiles, GroupCtl* ctl, bool rel,
                      bool multi, bool staged) {
  void* const fs[2][2][2] = {
      {{(void*)k_nlist<false, false, false>, (void*)k_nlist<false, false, true>},
       {(void*)k_nlist<false, true, false>, (void*)k_nlist<false, true, true>}},
      {{(void*)k_nlist<true, false, false>, (void*)k_nlist<true, false, true>},
       {(void*)k_nlist<true, true, false>, (void*)k_nlist<true, true, true>}}};
  void* f = fs[multi ? 1 : 0][rel ? 1 : 0][staged ? 1 : 0];
  KernelCall k = make_call(f, ntiles, CELLS_PER_TILE * 32, 0);
  put(k, d); put(k, tl); put(k, ctl);
  return k;
}

}  // namespace gbmd

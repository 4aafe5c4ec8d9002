// sort_core.cuh -- the pieces of the cell sort, per particle or per bin, shared by the
// rebuild kernels (k_lists.cu) and the team kernel (k_team.cuh): cell of a particle and
// histogram, scatter into the bins, order inside a bin, and the re-sort of the particle
// arrays.  `qv` is the position shadow of the current step.
#pragma once
#include "launch.cuh"

namespace gbmd {

// Morton code of the top 10 bits of each fixed-point coordinate (on [0, 2^32))
__device__ __forceinline__ unsigned spread10(unsigned v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}
__device__ __forceinline__ unsigned fine_morton(const int4& q) {
  return spread10(((unsigned)q.x ^ 0x80000000u) >> 22) |
         (spread10(((unsigned)q.y ^ 0x80000000u) >> 22) << 1) |
         (spread10(((unsigned)q.z ^ 0x80000000u) >> 22) << 2);
}

// ---- binning + histogram ----
// the particle's sort bin, kept with its Morton code
__device__ __forceinline__ int bin_of(const SysDev& s, const int4* qv, int i) {
  const int4 q = qv[i];
  const int cx = cell_of_fixed(q.x, s.nc[0]);
  const int cy = cell_of_fixed(q.y, s.nc[1]);
  const int cz = cell_of_fixed(q.z, s.nc[2]);
  // the tree list sorts type-major (each type's particles contiguous, in cell order);
  // inside a bin every list orders by the particle's own Morton code
  const int r = s.lin2rank[(cz * s.nc[1] + cy) * s.nc[0] + cx] + (s.tree ? q.w * s.ncells : 0);
  s.key[i] = r;
  s.fkey[i] = fine_morton(q);
  return r;
}
__device__ __forceinline__ void bin_one(const SysDev& s, const int4* qv, int i) {
  const int r = bin_of(s, qv, i);
  // consecutive particles mostly share a bin: one atomic per distinct bin of the warp
  const unsigned am = __activemask();
  const unsigned peers = __match_any_sync(am, r);
  if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&s.cell_cnt[r], __popc(peers));
}

// The same, and the particle into the bin's bucket of `cap` entries at the place the
// histogram's atomic gives it; false: the bucket is full.
__device__ __forceinline__ bool bin_bucket(const SysDev& s, const int4* qv, int i, int* bucket,
                                           int cap) {
  const int r = bin_of(s, qv, i);
  const int lane = threadIdx.x & 31;
  const unsigned am = __activemask();
  const unsigned peers = __match_any_sync(am, r);
  const int leader = __ffs(peers) - 1;
  int at = 0;
  if (lane == leader) at = atomicAdd(&s.cell_cnt[r], __popc(peers));
  at = __shfl_sync(am, at, leader) + __popc(peers & ((1u << lane) - 1u));
  if (at < cap) bucket[(size_t)r * cap + at] = i;
  return at < cap;
}

// ---- scatter particle indices into their cells (unordered within a cell) ----
// one atomic per distinct bin of the warp; the peers take consecutive slots after
// their leader's (the order inside a bin is fixed later)
__device__ __forceinline__ void scatter_one(const SysDev& s, int i) {
  const int r = s.key[i];
  const int lane = threadIdx.x & 31;
  const unsigned am = __activemask();
  const unsigned peers = __match_any_sync(am, r);
  const int leader = __ffs(peers) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(&s.cell_cursor[r], __popc(peers));
  base = __shfl_sync(am, base, leader);
  s.members_tmp[base + __popc(peers & ((1u << lane) - 1u))] = i;
}

// a position shadow with the particle's index beside its type: w = j | type << 30
__device__ __forceinline__ int4 with_index(const int4& q, int j) {
  return make_int4(q.x, q.y, q.z, (int)((unsigned)j | (unsigned)q.w << CPOS_TYPE_SHIFT));
}

// ---- sort one bin's members (one warp) -> a deterministic order ----
// By (fine Morton code, index), so that consecutive members of a bin are spatial
// neighbours (the tree list's leaves; the force kernel's warps).
// The bin's n members, in any order at `src`, get the ranks b ..
__device__ __forceinline__ void cellsort_one(const SysDev& s, const int4* qv, const int* src, int b,
                                             int n) {
  const int lane = threadIdx.x & 31;
  // the sort key of member m: (fine code, index)
  auto key = [&](int v) -> unsigned long long {
    return ((unsigned long long)s.fkey[v] << 32) | (unsigned)v;
  };
  // the members' positions are copied in the same order: the list build then reads
  // a cell's candidates contiguously, however far the particles have drifted from
  // the order of the last re-sort
  if (n <= 32) {
    const int v = lane < n ? src[lane] : 0x7fffffff;
    const unsigned long long kv = lane < n ? key(v) : ~0ull;
    int rk = 0;
    for (int k = 0; k < 32; ++k) rk += __shfl_sync(0xffffffffu, kv, k) < kv;
    if (lane < n) {
      s.members[b + rk] = v;
      s.rmember[v] = b + rk;
      s.cpos[b + rk] = with_index(qv[v], v);
    }
  } else {   // 32 members against 32 at a time, every key read once per block of 32
    for (int m0 = 0; m0 < n; m0 += 32) {
      const int m = m0 + lane;
      const int v = m < n ? src[m] : 0x7fffffff;
      const unsigned long long kv = m < n ? key(v) : ~0ull;
      int rk = 0;
      for (int k0 = 0; k0 < n; k0 += 32) {
        const unsigned long long ko =
            k0 == m0 ? kv : k0 + lane < n ? key(src[k0 + lane]) : ~0ull;
        for (int k = 0; k < 32; ++k) rk += __shfl_sync(0xffffffffu, ko, k) < kv;
      }
      if (m < n) {
        s.members[b + rk] = v;
        s.rmember[v] = b + rk;
        s.cpos[b + rk] = with_index(qv[v], v);
      }
    }
  }
}

// ---- re-sort: gather every per-particle array into cell order ----
__device__ __forceinline__ void permute_one(const SysDev& s, const int4* qv, int k) {
  const int n = s.n;
  const int o = s.members[k];
  for (int a = 0; a < 3; ++a) {
    s.x_alt[a * n + k] = s.x[a * n + o];
    s.v_alt[a * n + k] = s.v[a * n + o];
    s.img_alt[a * n + k] = s.img[a * n + o];
  }
  s.type_alt[k] = s.type[o];
  s.tag_alt[k] = s.tag[o];
  s.q_alt[k] = qv[o];
}

__device__ __forceinline__ void copyback_one(const SysDev& s, long long step, int k) {
  const int n = s.n;
  double xr[3];   // in units of L / 2^32
  for (int a = 0; a < 3; ++a) {
    const double xq = s.x_alt[a * n + k];
    s.x[a * n + k] = xq;
    s.v[a * n + k] = s.v_alt[a * n + k];
    s.img[a * n + k] = s.img_alt[a * n + k];
    xr[a] = xq;
  }
  const int ty = s.type_alt[k];
  s.type[k] = ty;
  const int tg = s.tag_alt[k];
  s.tag[k] = tg;
  s.rtag[tg] = k;
  q_at(s, step)[k] = s.q_alt[k];
  s.members[k] = k;
  s.rmember[k] = k;
  s.cpos[k] = with_index(s.q_alt[k], k);
  if (s.precision == GBMD_FP64)
    p64_at(s, step)[k] = fix_position(s, xr[0], xr[1], xr[2], ty);
}

}  // namespace gbmd

// nlist_split.cuh -- the cell list's neighbour rows for systems with few cells.
//
// The builder of the large systems (k_nlist) gives a cell to one warp, a lane to each
// of its particles: 9 to 14 thousand warp instructions per cell one after another.
// With fewer cells than the chip has warps that chain is the build's time (N = 20,000:
// 729 warps on 608 schedulers, 45 us; N = 500: eight warps, 104 us).  Here four warps
// share a cell.  They stage its stencil's candidates once, each a quarter of the
// stream, culled against the bounding box of the cell's particles, into shared memory;
// then each warp takes eight particles, four lanes each, culls the staged candidates
// again against its eight particles' smaller box and tests a chunk of 32 with eight
// candidates per lane.  The instructions per cell are about k_nlist's, the chain a
// quarter of it.
//
// The rows are the same: candidates in (stencil cell, member) order, the same decision
// (FP32 on the fixed-point difference, FP64 within the band) and the same order of the
// hits, so either builder may serve a system.
#pragma once
#include "launch.cuh"
#include "nlist_core.cuh"

namespace gbmd {

constexpr int NS_W = 4;    // warps sharing a cell
constexpr int NS_T = NS_W * 32;
constexpr int NS_P = 8;    // particles of a warp
constexpr int NS_C = 4;    // lanes of a particle
constexpr int NS_K = 32 / NS_C;   // candidates of a chunk that a lane tests
constexpr int NS_SEG = 256;       // staged candidates of a warp's quarter
constexpr int NS_CAP = NS_W * NS_SEG;   // candidates staged at a time (before culling)

// one warp's chunk ring: candidates 2m and 2m + 1 interleaved as cxy[m] = (x, x', y,
// y'), czt[m] = (z, z', t, t') (as k_nlist's), and j | type << 30; self[p]: the ring
// position of particle p's own candidate
struct SplitRing {
  float4 cxy[32], czt[32];
  int cj[64];
  int self[NS_P];
};
// what the warps of a cell share
struct SplitCell {
  float4 cand[NS_CAP];   // x, y, z relative to the cell's centre (raw fixed point with
                         // fewer than 3 cells on an axis), j | type << 30
  int at[NS_CAP];        // the candidate's member rank
  int kept[NS_W];        // candidates in each quarter
  float box[NS_W][6];
  SplitRing ring[NS_W];
};
// r_list^2 (1 - band) and, for the FP64 decision, r_list^2 per type pair
struct SplitTable {
  float lo[MAXT2];
  double rl2[MAXT2];
  float cull2;   // culling radius^2: the largest r_list with band and margin
};

// every thread of the block calls it; followed by a __syncthreads
__device__ __forceinline__ void split_table(const SysDev& s, SplitTable& t) {
  const int nt = s.ntypes;
  if ((int)threadIdx.x < nt * nt) {
    t.lo[threadIdx.x] = s.pf[threadIdx.x].rl2 * (1.0f - NL_BAND);
    t.rl2[threadIdx.x] = s.pd[threadIdx.x].rl2;
  }
  if (threadIdx.x == 0) {
    float hi = 0.0f;
    for (int k = 0; k < nt * nt; ++k) hi = fmaxf(hi, s.pf[k].rl2 * (1.0f + NL_BAND));
    t.cull2 = hi * (1.0f + NL_CULL_MARGIN);
  }
}

// a barrier over the NS_T threads that share a cell (`group` of the block; barrier 0 is
// the block's own)
__device__ __forceinline__ void split_sync(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(NS_T) : "memory");
}

// The rows of the particles 32 sub .. 32 sub + 31, 32 (sub + nsub) .., of cell rank r.
// Adds the neighbours found to nb_sum; returns the longest row that passed the
// capacity (0: none).  The NS_T threads of the block's group `bar` call it
// together; `sc` is theirs, free on entry once they have all arrived.
template <bool MULTI>
__device__ __forceinline__ int nlist_split(const SysDev& s, int r, int sub, int nsub, int bar,
                                           SplitCell& sc, const SplitTable& tab,
                                           unsigned long long& nb_sum) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & (NS_W - 1);
  const int p = lane / NS_C, c4 = lane % NS_C;
  const int b = s.cell_start[r], e = s.cell_start[r + 1];
  constexpr int PASS = NS_W * NS_P;
  if (b + PASS * sub >= e) return 0;   // uniform over the group
  SplitRing& ring = sc.ring[w];
  const int nt = s.ntypes;
  const int nc0 = s.nc[0], nc1 = s.nc[1], nc2 = s.nc[2];
  const int lin = s.rank2lin[r];
  const int cx = lin % nc0, cy = (lin / nc0) % nc1, cz = lin / (nc0 * nc1);
  // with 3 cells on every axis a coordinate relative to the cell's centre is already
  // the minimum image with respect to the cell's particles; with fewer the difference
  // is taken in fixed point per test and nothing is culled
  const bool rel = nc0 >= 3 && nc1 >= 3 && nc2 >= 3;
  const int ox = rel ? cell_centre_fixed(cx, nc0) : 0, oy = rel ? cell_centre_fixed(cy, nc1) : 0,
            oz = rel ? cell_centre_fixed(cz, nc2) : 0;
  const float fs0 = s.fscale[0], fs1 = s.fscale[1], fs2 = s.fscale[2];
  const int lo0 = nc0 >= 3 ? -1 : 0, n0 = nc0 >= 3 ? 3 : nc0;
  const int lo1 = nc1 >= 3 ? -1 : 0, n1 = nc1 >= 3 ? 3 : nc1;
  const int lo2 = nc2 >= 3 ? -1 : 0, n2 = nc2 >= 3 ? 3 : nc2;
  const int nsc = n0 * n1 * n2;
  int sc_start = 0, sc_cnt = 0;
  if (lane < nsc) {
    const int x = (cx + lo0 + lane % n0 + nc0) % nc0, y = (cy + lo1 + (lane / n0) % n1 + nc1) % nc1,
              z = (cz + lo2 + lane / (n0 * n1) + nc2) % nc2;
    const int nr = s.lin2rank[(z * nc1 + y) * nc0 + x];
    sc_start = s.cell_start[nr];
    sc_cnt = s.cell_start[nr + 1] - sc_start;
  }
  int incl = sc_cnt;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int excl = incl - sc_cnt;
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  const int cap = s.cap;
  const size_t group = (size_t)s.nl_stride * 4;   // entries of a slot group of the list
  int* const nl = s.nl;
  const int4* cpos = s.cpos;
  const float km1 = 2.0f * NL_BAND / (1.0f - NL_BAND);
  const bool two = !MULTI || nt <= 2;
  const float cull2 = tab.cull2;
  auto rel3 = [&](const int4& q) {
    return make_float3((float)min_image_fixed(q.x, ox) * fs0, (float)min_image_fixed(q.y, oy) * fs1,
                       (float)min_image_fixed(q.z, oz) * fs2);
  };

  // the bounding box of the cell's particles (of every pass)
  split_sync(bar);   // the previous cell's staging has been read
  float box[6];
  {
    float lo[3] = {3e38f, 3e38f, 3e38f}, hi[3] = {-3e38f, -3e38f, -3e38f};
    for (int m = b + (w * 32 + lane); m < e; m += NS_T) {
      const float3 a = rel3(cpos[m]);
      lo[0] = fminf(lo[0], a.x); hi[0] = fmaxf(hi[0], a.x);
      lo[1] = fminf(lo[1], a.y); hi[1] = fmaxf(hi[1], a.y);
      lo[2] = fminf(lo[2], a.z); hi[2] = fmaxf(hi[2], a.z);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo[k] = warp_min(lo[k]);
      hi[k] = warp_max(hi[k]);
    }
    if (lane == 0)
      for (int k = 0; k < 3; ++k) {
        sc.box[w][2 * k] = lo[k];
        sc.box[w][2 * k + 1] = hi[k];
      }
    split_sync(bar);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      float v = sc.box[0][k];
      for (int q = 1; q < NS_W; ++q) v = (k & 1) ? fmaxf(v, sc.box[q][k]) : fminf(v, sc.box[q][k]);
      box[k] = v;
    }
  }
  // candidates [base, base + NS_CAP) of the flattened stream into the staging area:
  // this warp's quarter, in order, those that can reach the cell's particles
  auto stage = [&](int base) {
    const int end = min(total, base + NS_CAP);
    const int quarter = ((end - base + NS_W * 32 - 1) / (NS_W * 32)) * 32;   // <= NS_SEG
    const int q0 = base + w * quarter, q1 = min(end, q0 + quarter);
    int kept = 0;
    for (int c0 = q0; c0 < q1; c0 += 32) {
      const int c = c0 + lane;
      int lo = 0;   // the stencil cell of candidate c
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int mid = lo + step;
        const int v = __shfl_sync(0xffffffffu, excl, mid & 31);
        if (mid < nsc && c >= v) lo = mid;
      }
      const int at = __shfl_sync(0xffffffffu, sc_start - excl, lo) + c;
      bool keep = c < q1;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (keep) {
        const int4 q = cpos[at];
        if (rel) {
          const float3 a = rel3(q);
          const float gx = gap_to(a.x, box[0], box[1]), gy = gap_to(a.y, box[2], box[3]),
                      gz = gap_to(a.z, box[4], box[5]);
          keep = fmaf(gz, gz, fmaf(gy, gy, gx * gx)) < cull2;
          v = make_float4(a.x, a.y, a.z, __int_as_float(q.w));
        } else {
          v = make_float4(__int_as_float(q.x), __int_as_float(q.y), __int_as_float(q.z),
                          __int_as_float(q.w));
        }
      }
      const unsigned kb = __ballot_sync(0xffffffffu, keep);
      if (keep) {
        const int sl = w * NS_SEG + kept + __popc(kb & ((1u << lane) - 1u));
        sc.cand[sl] = v;
        sc.at[sl] = at;
      }
      kept += __popc(kb);
    }
    if (lane == 0) sc.kept[w] = kept;
  };

  const bool whole = total <= NS_CAP;   // the stream fits: staged once for every pass
  if (whole) {
    stage(0);
    split_sync(bar);
  }
  int over = 0;
  for (int g0 = b + PASS * sub; g0 < e; g0 += PASS * nsub) {   // uniform over the group
    const int g = g0 + w * NS_P;
    const bool valid = g + p < e;
    const int4 qi = valid ? cpos[g + p] : make_int4(0, 0, 0, 0);
    const int i = qi.w & ((1 << NL_TYPE_SHIFT) - 1), ti = (int)((unsigned)qi.w >> NL_TYPE_SHIFT);
    const float3 a = rel3(qi);
    const float2 nX = make_float2(-a.x, -a.x), nY = make_float2(-a.y, -a.y), nZ = make_float2(-a.z, -a.z);
    const float bx0 = warp_min(valid ? a.x : 3e38f), bx1 = warp_max(valid ? a.x : -3e38f);
    const float by0 = warp_min(valid ? a.y : 3e38f), by1 = warp_max(valid ? a.y : -3e38f);
    const float bz0 = warp_min(valid ? a.z : 3e38f), bz1 = warp_max(valid ? a.z : -3e38f);
    const int pt = MULTI ? ti * nt : 0;
    const float lo_0 = valid ? tab.lo[pt] : -1.0f;   // an idle lane never keeps
    const float lo_1 = valid && MULTI ? tab.lo[pt + min(1, nt - 1)] : lo_0;
    const float2 nl0 = make_float2(-lo_0, -lo_0), ndl = make_float2(lo_0 - lo_1, lo_0 - lo_1);
    const float2 k2 = make_float2(km1, km1);
    int* const row = nl + (size_t)i * 4;
    int cnt = 0;
    int fill = 0, tested = 0;
    if (lane < NS_P) ring.self[lane] = -1;
    __syncwarp();

    // -(r_list^2 (1 - band)) of this particle with the candidate of word `cw`
    auto neg_lo = [&](int cw) -> float {
      return valid ? -tab.lo[pt + (int)((unsigned)cw >> NL_TYPE_SHIFT)] : 1.0f;
    };
    // the chunk at ring slots hb .. hb + 31: this lane takes NS_K of them
    auto test = [&](int hb) {
      const int h0 = hb + NS_K * c4;
      unsigned mlo = 0u, mhi = 0u;   // candidate h0 + k at bit NS_K - 1 - k
#pragma unroll
      for (int k = 0; k < NS_K; k += 2) {
        const float4 A = ring.cxy[(h0 + k) >> 1], B = ring.czt[(h0 + k) >> 1];
        float2 nlo;
        if (!MULTI) nlo = nl0;
        else if (two) nlo = __ffma2_rn(make_float2(B.z, B.w), ndl, nl0);
        else nlo = make_float2(neg_lo(ring.cj[h0 + k]), neg_lo(ring.cj[h0 + k + 1]));
        float2 dx, dy, dz;
        if (rel) {
          dx = __fadd2_rn(make_float2(A.x, A.y), nX);
          dy = __fadd2_rn(make_float2(A.z, A.w), nY);
          dz = __fadd2_rn(make_float2(B.x, B.y), nZ);
        } else {
          auto d1 = [](int q, float x, float f) { return (float)min_image_fixed(q, __float_as_int(x)) * f; };
          dx = make_float2(d1(qi.x, A.x, fs0), d1(qi.x, A.y, fs0));
          dy = make_float2(d1(qi.y, A.z, fs1), d1(qi.y, A.w, fs1));
          dz = make_float2(d1(qi.z, B.x, fs2), d1(qi.z, B.y, fs2));
        }
        float2 d = __ffma2_rn(dx, dx, nlo);
        d = __ffma2_rn(dy, dy, d);
        d = __ffma2_rn(dz, dz, d);                  // r^2 - lo
        const float2 dh = __ffma2_rn(nlo, k2, d);   // r^2 - hi
        mlo = push_sign(push_sign(mlo, d.x), d.y);
        mhi = push_sign(push_sign(mhi, dh.x), dh.y);
      }
      const int rs = ring.self[p] - tested - NS_K * c4;
      unsigned keep = (1u << NS_K) - 1u;
      if (rs >= 0 && rs < NS_K) keep &= ~((1u << (NS_K - 1)) >> rs);
      const int left = fill - tested - NS_K * c4;   // slots past the stream's end
      if (left < NS_K) keep &= left > 0 ? ~((1u << (NS_K - left)) - 1u) : 0u;
      mhi &= keep;
      unsigned band = mhi & ~mlo;
      while (band) {
        const int bit = 31 - __clz(band);
        band &= ~(1u << bit);
        const int cw = ring.cj[h0 + NS_K - 1 - bit];
        const int pr = MULTI ? pt + (int)((unsigned)cw >> NL_TYPE_SHIFT) : 0;
        if (!exact_within(s, i, cw & ((1 << NL_TYPE_SHIFT) - 1), tab.rl2[pr])) mhi &= ~(1u << bit);
      }
      // the particle's hits of the chunk over its four lanes, in candidate order
      unsigned all = mhi << (NS_K * (NS_C - 1 - c4));
      all |= __shfl_xor_sync(0xffffffffu, all, 1);
      all |= __shfl_xor_sync(0xffffffffu, all, 2);
      int at = cnt + (c4 ? __popc(all >> (NS_K * (NS_C - c4))) : 0);
      while (mhi) {
        const int bit = 31 - __clz(mhi);
        mhi &= ~(1u << bit);
        const int j = ring.cj[h0 + NS_K - 1 - bit] & ((1 << NL_TYPE_SHIFT) - 1);
        if (at < cap) row[(size_t)(at >> 2) * group + (at & 3)] = j;
        ++at;
      }
      cnt += __popc(all);
    };
    // the staged candidates through this warp's ring
    auto process = [&]() {
      const int k0 = sc.kept[0], k1 = k0 + sc.kept[1], k2n = k1 + sc.kept[2], k3 = k2n + sc.kept[3];
      for (int cb = 0; cb < k3; cb += 32) {
        const int c = cb + lane;
        const int sl = c < k0 ? c : c < k1 ? c - k0 + NS_SEG : c < k2n ? c - k1 + 2 * NS_SEG
                                                                      : c - k2n + 3 * NS_SEG;
        bool keep = c < k3;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        int at = 0;
        if (keep) {
          v = sc.cand[sl];
          at = sc.at[sl] - g;
        }
        if (rel) {
          const float gx = gap_to(v.x, bx0, bx1), gy = gap_to(v.y, by0, by1), gz = gap_to(v.z, bz0, bz1);
          keep = keep && fmaf(gz, gz, fmaf(gy, gy, gx * gx)) < cull2;
        }
        const unsigned kb = __ballot_sync(0xffffffffu, keep);
        if (keep) {
          const int pos = fill + __popc(kb & ((1u << lane) - 1u)), ps = pos & 63;
          float* f = reinterpret_cast<float*>(&ring.cxy[ps >> 1]) + (ps & 1);
          float* q = reinterpret_cast<float*>(&ring.czt[ps >> 1]) + (ps & 1);
          const unsigned cw = __float_as_uint(v.w);
          f[0] = v.x;
          f[2] = v.y;
          q[0] = v.z;
          if (MULTI) q[2] = (cw >> NL_TYPE_SHIFT) & 1u ? 1.0f : 0.0f;
          ring.cj[ps] = (int)cw;
          if ((unsigned)at < (unsigned)NS_P) ring.self[at] = pos;
        }
        fill += __popc(kb);
        __syncwarp();
        if (fill - tested >= 32) {
          test(tested & 63);
          tested += 32;
        }
        __syncwarp();
      }
    };
    if (whole) {
      if (g < e) process();
    } else {
      for (int base = 0; base < total; base += NS_CAP) {
        split_sync(bar);   // the staging area has been read
        stage(base);
        split_sync(bar);
        if (g < e) process();
      }
    }
    if (fill > tested) test(tested & 63);
    __syncwarp();
    if (valid && c4 == 0) {
      s.nn[i] = cnt < cap ? cnt : cap;
      s.q_build[i] = make_int4(qi.x, qi.y, qi.z, ti);
      nb_sum += (unsigned long long)cnt;
      if (cnt > cap) over = max(over, cnt);
    }
  }
  return over;
}

}  // namespace gbmd

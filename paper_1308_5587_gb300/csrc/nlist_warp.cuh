// nlist_warp.cuh -- the cell list's neighbour rows of one cell, built by one warp (the
// builder of systems with many cells; nlist_split.cuh has the other).
#pragma once
#include "launch.cuh"
#include "nlist_core.cuh"

namespace gbmd {

// ---- neighbour list: one warp per cell ----
// Lanes are the cell's particles (up to 32 at a time).  The candidates -- the
// members of the stencil cells in (dz, dy, dx) cell order and member order within
// a cell, flattened into one stream, their positions and indices read from the copy in
// cell order that the cell sort wrote -- pass through a per-warp shared-memory buffer
// 32 at a time, each converted once into FP32 coordinates relative to the centre
// of the warp's cell (the fixed-point difference takes care of the periodic wrap);
// the next chunk is loaded while the current one is tested.  Every lane then tests the
// broadcast candidate against its own particle with packed FP32x2 arithmetic (no
// integer work per test), so each row holds its neighbours in (stencil cell, member)
// order.  Candidates within a relative band of 1e-5 of r_list^2 are decided in FP64 as
// the definition does (the FP32 error is below 2e-6 relative).
//
// With at least 3 cells per axis (REL) each chunk is first culled: a candidate
// farther than the largest r_list from the bounding box of the warp's particles
// cannot be anyone's neighbour, and the survivors are compacted (at KA density
// 44% of the stencil lies outside that reach).
//
// The kernel is bound by instruction issue, so a hit must cost few instructions.  The
// test of a chunk appends as it goes: a predicated store of the candidate's index into
// the lane's column of a shared-memory buffer and a predicated step of its pointer, no
// loop over hit masks (whose trips follow the lane with the most hits and cost ~20
// instructions each).  The buffer empties into the row four entries to a 16-byte
// store.  A chunk with a candidate in the band of some lane, ~3% of them, is tested
// again with hit masks.  LJ fluid, N = 200,000, at creation: 118 us and 83.6 M warp
// instructions with masks kept per chunk and appended in a deferred loop, 107 us and 71.5 M
// with the buffer; KA 10^6: 656 us and 463 M, 583 us and 400 M.
//
// SLOTS: hits of a lane that wait, 32 of a chunk and up to SLOTS - 32 before.  More slots,
// fewer and fuller flushes; the team kernel takes fewer, so that its force phase keeps
// the L1 (shared memory and L1 share the SM's 256 KB).
constexpr int NL_SLOTS = 56, NL_SLOTS_TEAM = 40;
// With at least 3 cells on every axis, a candidate's coordinate relative to the cell
// centre, taken in [-L/2, L/2), is already its minimum image with respect to every
// particle of the cell (|d| < r_list <= w and the particle lies within w/2 of the
// centre).  With 1 or 2 cells on an axis a neighbour may sit on either side, so such
// a system keeps fixed-point coordinates and takes the minimum image per test.  The
// REL instance serves launches whose systems all have 3 cells per axis; the other
// decides per system.

// a warp's shared memory
template <bool STAGED, int SLOTS = NL_SLOTS>
struct WarpRing {
  // the chunk of candidates: x, y, z (relative to the cell centre; raw fixed point
  // without REL) and the type as 0/1, candidates 2m and 2m + 1 interleaved as
  // cxy[m] = (x, x', y, y') and czt[m] = (z, z', t, t') so that a pair loads as two
  // 16-byte words of FP32x2 operands; j; and j | type << 30
  float4 cxy[32], czt[32];
  int4 cj[16];
  int cjs[64];
  int hits[SLOTS][32];        // a lane's hits that are not in its row yet
  double rl2d[MAXT2];
  float thr_lo[MAXT2], thr_hi[MAXT2];   // r_list^2 (1 -+ band) per type pair
  float wbox[6];                 // the pass's bounding box (culling)
  int cand_l[STAGED ? 64 : 1];   // window-local index
};

// Where d < 0 (SELF: and `other` is not 0), store j at shared address `at` and step to
// the lane's next slot: predicated instructions, no branch.  (No memory clobber, or the
// loads of the next candidates would wait; the caller puts one after the chunk.)
template <bool SELF>
__device__ __forceinline__ void append_if(unsigned& at, int j, float d, int other) {
  if constexpr (SELF)
    asm volatile("{ .reg .pred p, q; setp.ne.s32 q, %3, 0; setp.lt.and.f32 p, %2, 0f00000000, q;\n\t"
                 "@p st.shared.s32 [%0], %1;\n\t@p add.u32 %0, %0, 128; }"
                 : "+r"(at) : "r"(j), "f"(d), "r"(other));
  else
    asm volatile("{ .reg .pred p; setp.lt.f32 p, %2, 0f00000000;\n\t"
                 "@p st.shared.s32 [%0], %1;\n\t@p add.u32 %0, %0, 128; }"
                 : "+r"(at) : "r"(j), "f"(d));
}

// The rows of cell rank r's particles.  Adds the neighbours found to nb_sum; returns
// the longest row that passed the capacity (0: none).  Every lane of the warp calls it.
template <bool MULTI, bool REL, bool STAGED, int SLOTS>
__device__ __forceinline__ int nlist_cell(const SysDev& s, int r, WarpRing<STAGED, SLOTS>& sm,
                                          unsigned long long& nb_sum) {
  const int lane = threadIdx.x & 31;
  const int nt = s.ntypes;
  int over = 0;
  // STAGED: some member of the group may use the staged force path (decided per
  // system below); otherwise none does
  const bool staged = STAGED && s.staged != 0;   // then every axis has >= 4 cells
  float hi_max = 0.0f;
  for (int k = lane; k < nt * nt; k += 32) {
    const float rl2 = s.pf[k].rl2;
    sm.thr_lo[k] = rl2 * (1.0f - NL_BAND);
    sm.thr_hi[k] = rl2 * (1.0f + NL_BAND);
    sm.rl2d[k] = s.pd[k].rl2;
    hi_max = fmaxf(hi_max, sm.thr_hi[k]);
  }
  hi_max = warp_max(hi_max);
  // culling radius^2 of a chunk (the largest r_list, with margin)
  const float cull2 = hi_max * (1.0f + NL_CULL_MARGIN);
  // r^2 - hi = (r^2 - lo) - (kappa - 1) lo, kappa = (1 + band) / (1 - band)
  const float km1 = 2.0f * NL_BAND / (1.0f - NL_BAND);
  // the widest band: r^2 - lo of a candidate in the band lies in [0, wb) (a little wider
  // than the widest pair's, so rounding loses none)
  const unsigned wb = __float_as_uint(hi_max * (2.1f * NL_BAND));
  const int nc0 = s.nc[0], nc1 = s.nc[1], nc2 = s.nc[2];
  const int lin = s.rank2lin[r];
  const int cx = lin % nc0, cy = (lin / nc0) % nc1, cz = lin / (nc0 * nc1);
  const int ox = cell_centre_fixed(cx, nc0), oy = cell_centre_fixed(cy, nc1),
            oz = cell_centre_fixed(cz, nc2);
  const float fs0 = s.fscale[0], fs1 = s.fscale[1], fs2 = s.fscale[2];
  // distinct neighbour-cell offsets per axis (fewer than 3 cells: no duplicates)
  const int lo0 = nc0 >= 3 ? -1 : 0, n0 = nc0 >= 3 ? 3 : nc0;
  const int lo1 = nc1 >= 3 ? -1 : 0, n1 = nc1 >= 3 ? 3 : nc1;
  const int lo2 = nc2 >= 3 ? -1 : 0, n2 = nc2 >= 3 ? 3 : nc2;
  const int nsc = n0 * n1 * n2;   // <= 27
  // REL: every system of the launch has >= 3 cells per axis; otherwise each system
  // takes the relative-coordinate path when it has them (warp-uniform: a warp is one
  // cell of one system), so a batch with one small member builds the others fast
  const bool rel = REL || (nc0 >= 3 && nc1 >= 3 && nc2 >= 3);
  const int own_sc = -lo0 + n0 * (-lo1 + n1 * -lo2);   // the cell's own stencil slot
  int sc_start = 0, sc_cnt = 0, sc_woff = 0;
  if (lane < nsc) {
    const int dx = lo0 + lane % n0, dy = lo1 + (lane / n0) % n1, dz = lo2 + lane / (n0 * n1);
    const int x = (cx + dx + nc0) % nc0, y = (cy + dy + nc1) % nc1, z = (cz + dz + nc2) % nc2;
    const int nr = s.lin2rank[(z * nc1 + y) * nc0 + x];
    sc_start = s.cell_start[nr];
    sc_cnt = s.cell_start[nr + 1] - sc_start;
    if (staged) {   // this stencil cell's place in the block's 4x4x4 window
      const int blk = ((cz >> 1) * s.nb[1] + (cy >> 1)) * s.nb[0] + (cx >> 1);
      const int wi = (((cz & 1) + 1 + dz) * 4 + ((cy & 1) + 1 + dy)) * 4 + ((cx & 1) + 1 + dx);
      sc_woff = s.blk_win[(size_t)blk * WIN_CELLS + wi].y;
    }
  }
  int incl = sc_cnt;   // inclusive prefix of the stencil cells' sizes
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int excl = incl - sc_cnt;
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  const int b = s.cell_start[r], e = s.cell_start[r + 1];
  const int cap = s.cap;
  const int4* cpos = s.cpos;   // member m's position, index and type (from the cell sort)
  const bool two = !MULTI || nt <= 2;
  constexpr int JMASK = (1 << NL_TYPE_SHIFT) - 1;
  __syncwarp();

  auto put_cand = [&](int sl, float x, float y, float z, float t) {
    float* a = reinterpret_cast<float*>(&sm.cxy[sl >> 1]) + (sl & 1);
    float* c = reinterpret_cast<float*>(&sm.czt[sl >> 1]) + (sl & 1);
    a[0] = x;
    a[2] = y;
    c[0] = z;
    if (MULTI) c[2] = t;
  };
  // component a (0 x, 1 y, 2 z) of slot sl
  auto cand_comp = [&](int sl, int a) -> float {
    const float* q = reinterpret_cast<const float*>(a < 2 ? &sm.cxy[sl >> 1] : &sm.czt[sl >> 1]);
    return q[(a == 1 ? 2 : 0) + (sl & 1)];
  };

  // candidate c of the flattened stream into registers (every lane runs every
  // shuffle); written to the chunk arrays once the previous chunk is done
  int4 nq = make_int4(0, 0, 0, 0);   // w = j | type << 30 (types 2, 3 set the sign bit)
  bool nempty = true;                // past the end of the stream
  int nloc = 0;
  const int sc_shift = sc_start - excl;
  auto fetch = [&](int c) {
    int lo = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int mid = lo + step;
      const int v = __shfl_sync(0xffffffffu, excl, mid & 31);
      if (mid < nsc && c >= v) lo = mid;
    }
    const int at = __shfl_sync(0xffffffffu, sc_shift, lo) + c;
    if (STAGED) nloc = __shfl_sync(0xffffffffu, sc_woff - excl, lo) + c;
    nempty = c >= total;
    if (!nempty) nq = cpos[at];
  };

  for (int ibase = b; ibase < e; ibase += 32) {
    const bool valid = ibase + lane < e;
    const int4 qi = valid ? cpos[ibase + lane] : make_int4(0, 0, 0, 0);
    const int i = valid ? qi.w & JMASK : -1;
    const int ti = (int)((unsigned)qi.w >> NL_TYPE_SHIFT);
    const float xi = (float)min_image_fixed(qi.x, ox) * fs0;
    const float yi = (float)min_image_fixed(qi.y, oy) * fs1;
    const float zi = (float)min_image_fixed(qi.z, oz) * fs2;
    const float2 nX = make_float2(-xi, -xi), nY = make_float2(-yi, -yi), nZ = make_float2(-zi, -zi);
    // the bounding box of this pass's particles (REL culling)
    // (kept in shared memory: read once per fetched chunk, they need no registers)
    {
      const float bx0 = warp_min(valid ? xi : 3e38f), bx1 = warp_max(valid ? xi : -3e38f);
      const float by0 = warp_min(valid ? yi : 3e38f), by1 = warp_max(valid ? yi : -3e38f);
      const float bz0 = warp_min(valid ? zi : 3e38f), bz1 = warp_max(valid ? zi : -3e38f);
      if (lane == 0) {
        sm.wbox[0] = bx0; sm.wbox[1] = bx1; sm.wbox[2] = by0;
        sm.wbox[3] = by1; sm.wbox[4] = bz0; sm.wbox[5] = bz1;
      }
      __syncwarp();
    }
    // An idle lane gets thresholds -1 (never keeps).  Two types: -lo for a type-0
    // candidate and its change for type 1 in registers; more types read the table.
    const int pt = MULTI ? ti * nt : 0;
    const float lo_0 = valid ? sm.thr_lo[pt] : -1.0f;
    const float lo_1 = valid && MULTI ? sm.thr_lo[pt + min(1, nt - 1)] : lo_0;
    const float2 nl0 = make_float2(-lo_0, -lo_0), ndl = make_float2(lo_0 - lo_1, lo_0 - lo_1);
    const int stride = s.nl_stride;
    const int i_row = valid ? i : 0;
    int cnt = 0;   // entries in the row
    const int m_row = ibase + lane;   // member rank (staged list rows)
    int* const nl = s.nl;
    unsigned short* nl16 = reinterpret_cast<unsigned short*>(nl);
    int4* const nl4 = reinterpret_cast<int4*>(nl) + i_row;
    // the particle's own place in the candidate stream (its cell is stencil cell
    // own_sc; a pass covers members ibase .. ibase + 31 of that cell)
    const int self_pos = __shfl_sync(0xffffffffu, excl, own_sc) + (ibase - b) + lane;

    // Hits of the 32 candidates at ring slots hb .. hb + 31: candidate k at bit 31 - k
    // of mlo (r^2 below lo: a neighbour) and mhi (below hi: a neighbour or within the
    // band).  The band is decided in FP64 first; then the hits are taken in candidate
    // order (the row does not depend on how r^2 was rounded).  Entries past the
    // capacity are counted, not stored.
    auto resolve_band = [&](unsigned mlo, unsigned mhi, int hb) -> unsigned {
      unsigned band = mhi & ~mlo;
      while (band) {
        const int k = __clz(band);
        band &= 0x7fffffffu >> k;
        const int cw = sm.cjs[hb + k];
        const int p = MULTI ? pt + (int)((unsigned)cw >> NL_TYPE_SHIFT) : 0;
        if (!exact_within(s, i, cw & JMASK, sm.rl2d[p])) mhi &= ~(0x80000000u >> k);
      }
      return mhi;
    };
    auto append_hits = [&](unsigned mlo, unsigned mhi, int hb) {
      mhi = resolve_band(mlo, mhi, hb);
      while (mhi) {
        const int k = __clz(mhi);
        mhi &= 0x7fffffffu >> k;
        if (cnt < cap) {
          if (staged) nl16[nl16_index(m_row, cnt, stride)] = (unsigned short)sm.cand_l[hb + k];
          else nl[nl_index(i_row, cnt, stride)] = sm.cjs[hb + k] & JMASK;
        }
        ++cnt;
      }
    };

    // the lane's waiting hits: slots 0 .. (column end - column) / 32 of its column
    int* const column = &sm.hits[0][lane];
    int* end = column;
    // whole groups of four into the row, the up to three left over to the front;
    // `last`: those too, the group filled up with its first entry (past the count)
    auto flush = [&](bool last) {
      const int c = (int)(end - column) >> 5;
      int* at = column;
      int4* row = nl4 + (size_t)(cnt >> 2) * stride;   // cnt is a multiple of 4 here
      for (int g = c >> 2; g > 0; --g) {
        const int4 v = make_int4(at[0], at[32], at[64], at[96]);
        if (cnt < cap) *row = v;
        row += stride;
        at += 128;
        cnt += 4;
      }
      const int left = c & 3;
      int j0 = 0, j1 = 0, j2 = 0;   // a full buffer ends behind its last slot: read what is left
      if (left > 0) j0 = at[0];
      if (left > 1) j1 = at[32];
      if (left > 2) j2 = at[64];
      if (last) {
        if (left && cnt < cap)
          *row = make_int4(j0, left > 1 ? j1 : j0, left > 2 ? j2 : j0, j0);
        cnt += left;
        end = column;
      } else {
        column[0] = j0;
        column[32] = j1;
        column[64] = j2;
        end = column + 32 * left;
      }
    };

    fetch(lane);
    if (rel) {
      // Kept candidates go into a ring of 64 slots in stream order; every time 32
      // are waiting they are tested together (a full, unrolled chunk), so culling
      // saves tests and not only stores.  The particle's own candidate is always
      // kept (it lies in the box); selfabs is its ring position.
      int fill = 0, tested = 0, selfabs = -1;
      // r^2 - lo of candidates k and k + 1 of the chunk at hb, and -lo
      auto diff = [&](int hb, int k, float2& nlo) -> float2 {
        const float4 A = sm.cxy[(hb + k) >> 1];
        const float4 B = sm.czt[(hb + k) >> 1];
        if (!MULTI) {
          nlo = nl0;
        } else if (two) {
          nlo = __ffma2_rn(make_float2(B.z, B.w), ndl, nl0);
        } else {
          const unsigned t0 = (unsigned)sm.cjs[hb + k] >> NL_TYPE_SHIFT;
          const unsigned t1 = (unsigned)sm.cjs[hb + k + 1] >> NL_TYPE_SHIFT;
          nlo = valid ? make_float2(-sm.thr_lo[pt + (t0 & 3)], -sm.thr_lo[pt + (t1 & 3)])
                      : make_float2(1.0f, 1.0f);
        }
        const float2 dx = __fadd2_rn(make_float2(A.x, A.y), nX);
        const float2 dy = __fadd2_rn(make_float2(A.z, A.w), nY);
        const float2 dz = __fadd2_rn(make_float2(B.x, B.y), nZ);
        float2 d = __ffma2_rn(dx, dx, nlo);
        d = __ffma2_rn(dy, dy, d);
        return __ffma2_rn(dz, dz, d);
      };
      auto masks = [&](int hb, int rs, unsigned& mlo, unsigned& mhi) {
        const float2 k2 = make_float2(km1, km1);
        mlo = mhi = 0u;
#pragma unroll 4
        for (int k = 0; k < 32; k += 2) {
          float2 nlo;
          const float2 d = diff(hb, k, nlo);
          const float2 dh = __ffma2_rn(nlo, k2, d);   // r^2 - hi
          mlo = push_sign(push_sign(mlo, d.x), d.y);
          mhi = push_sign(push_sign(mhi, dh.x), dh.y);
        }
        if (rs >= 0 && rs < 32) {
          mlo &= ~(0x80000000u >> rs);
          mhi &= ~(0x80000000u >> rs);
        }
      };
      // the chunk into the buffer; SELF: some lane's own candidate is in it (slot rs)
      auto append32 = [&](int hb, int rs, auto self) -> bool {
        constexpr bool SELF = decltype(self)::value;
        // the smallest r^2 - lo that is not negative: a float's bits order like unsigned
        // integers there, and a negative one's are above them all
        unsigned near = 0xffffffffu;
        unsigned at = (unsigned)__cvta_generic_to_shared(end);
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          const int4 j = sm.cj[(hb + k) >> 2];
          float2 nlo;
          const float2 d0 = diff(hb, k, nlo), d1 = diff(hb, k + 2, nlo);
          near = min(min(near, __float_as_uint(d0.x)), __float_as_uint(d0.y));
          near = min(min(near, __float_as_uint(d1.x)), __float_as_uint(d1.y));
          append_if<SELF>(at, j.x, d0.x, rs - k);
          append_if<SELF>(at, j.y, d0.y, rs - k - 1);
          append_if<SELF>(at, j.z, d1.x, rs - k - 2);
          append_if<SELF>(at, j.w, d1.y, rs - k - 3);
        }
        asm volatile("" ::: "memory");   // the buffer has been written
        if (near < wb) return true;      // its end stays: the chunk is tested again
        end += (at - (unsigned)__cvta_generic_to_shared(end)) >> 2;
        return false;
      };
      auto test32 = [&](int hb) {
        const int rs = selfabs - tested;
        if (staged) {
          unsigned mlo, mhi;
          masks(hb, rs, mlo, mhi);
          append_hits(mlo, mhi, hb);
          return;
        }
        const bool own = __any_sync(0xffffffffu, rs >= 0 && rs < 32);
        const bool band = own ? append32(hb, rs, std::true_type{}) : append32(hb, rs, std::false_type{});
        if (__any_sync(0xffffffffu, band)) {
          unsigned mlo, mhi;
          masks(hb, rs, mlo, mhi);
          if (band) {
            mhi = resolve_band(mlo, mhi, hb);
            while (mhi) {
              const int k = __clz(mhi);
              mhi &= 0x7fffffffu >> k;
              *end = sm.cjs[hb + k] & JMASK;
              end += 32;
            }
          }
          __syncwarp();
        }
        if (__any_sync(0xffffffffu, end > column + 32 * (SLOTS - 32))) flush(false);
      };
      for (int cb = 0; cb < total; cb += 32) {
        // relative coordinates; cull against the box and compact the survivors
        const float qx = (float)min_image_fixed(nq.x, ox) * fs0;
        const float qy = (float)min_image_fixed(nq.y, oy) * fs1;
        const float qz = (float)min_image_fixed(nq.z, oz) * fs2;
        const float gx = gap_to(qx, sm.wbox[0], sm.wbox[1]), gy = gap_to(qy, sm.wbox[2], sm.wbox[3]),
                    gz = gap_to(qz, sm.wbox[4], sm.wbox[5]);
        const bool keep = !nempty && fmaf(gz, gz, fmaf(gy, gy, gx * gx)) < cull2;
        const unsigned kb = __ballot_sync(0xffffffffu, keep);
        if (keep) {
          const int sl = (fill + __popc(kb & ((1u << lane) - 1u))) & 63;
          put_cand(sl, qx, qy, qz, (unsigned)nq.w >> NL_TYPE_SHIFT & 1u ? 1.0f : 0.0f);
          sm.cjs[sl] = nq.w;
          reinterpret_cast<int*>(sm.cj)[sl] = nq.w & JMASK;
          if (STAGED) sm.cand_l[sl] = nloc;
        }
        const int rs = self_pos - cb;
        if (rs >= 0 && rs < 32) selfabs = fill + __popc(kb & ((1u << rs) - 1u));
        fill += __popc(kb);
        __syncwarp();
        if (cb + 32 < total) fetch(cb + 32 + lane);   // in flight during the tests
        if (fill - tested >= 32) {
          test32(tested & 63);
          tested += 32;
        }
        __syncwarp();
      }
      if (fill > tested) {   // the last, partial chunk: pad it with far-away slots
        if (lane >= fill - tested) {
          const int sl = (tested + lane) & 63;
          put_cand(sl, 1e18f, 1e18f, 1e18f, 0.0f);
          sm.cjs[sl] = 0;
        }
        __syncwarp();
        test32(tested & 63);
        __syncwarp();
      }
      if (!staged) flush(true);
    } else {
      for (int cb = 0; cb < total; cb += 32) {
        put_cand(lane, __int_as_float(nq.x), __int_as_float(nq.y), __int_as_float(nq.z), 0.0f);
        sm.cjs[lane] = nq.w;
        if (STAGED) sm.cand_l[lane] = nloc;
        const int m = min(32, total - cb);
        __syncwarp();
        if (cb + 32 < total) fetch(cb + 32 + lane);   // in flight during the tests
        unsigned mlo = 0, mhi = 0;
        for (int k = 0; k < 32; ++k) {
          float r2 = 3e38f;
          int p = 0;
          if (k < m) {
            const float dx = (float)min_image_fixed(qi.x, __float_as_int(cand_comp(k, 0))) * fs0;
            const float dy = (float)min_image_fixed(qi.y, __float_as_int(cand_comp(k, 1))) * fs1;
            const float dz = (float)min_image_fixed(qi.z, __float_as_int(cand_comp(k, 2))) * fs2;
            r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const unsigned ct = (unsigned)sm.cjs[k] >> NL_TYPE_SHIFT;
            p = !MULTI ? 0 : two ? (int)(ct & 1) : (int)ct;
          }
          const float lo = valid ? sm.thr_lo[pt + p] : -1.0f;
          const float hi = valid ? sm.thr_hi[pt + p] : -1.0f;
          mlo = (mlo << 1) | (r2 < lo ? 1u : 0u);
          mhi = (mhi << 1) | (r2 < hi ? 1u : 0u);
        }
        const int rs = self_pos - cb;
        if (rs >= 0 && rs < 32) {
          mlo &= ~(0x80000000u >> rs);
          mhi &= ~(0x80000000u >> rs);
        }
        append_hits(mlo, mhi, 0);
        __syncwarp();
      }
    }
    if (valid) {
      s.nn[i] = cnt < cap ? cnt : cap;
      s.q_build[i] = make_int4(qi.x, qi.y, qi.z, ti);
      if (cnt > cap) over = max(over, cnt);
      nb_sum += (unsigned long long)cnt;
    }
  }
  return over;
}

}  // namespace gbmd

// k_team.cuh -- many steps of one system in one launch, by a team of thread blocks that
// stay resident: forces, integration, the rebuild decision and the whole list rebuild,
// with a barrier of the team (team_core.cuh) between the phases.
//
// Why: the graph of a step is one kernel and a conditional node with the rebuild's
// kernels.  Evaluating that node costs ~13 us a step (64k particles, mixed: 18.8 us for
// steps without the nodes, 32.6 us with them), a launch ~2 us, and a rebuild seven
// launches; in a batch, where some member rebuilds at nearly every step, every member
// waits for the whole chain.  A team needs one barrier a step (NVT: two) and three a rebuild
// (a re-sort two more, a bucket that ran over two more), and each system goes at its own pace.
//
// Blocks keep contiguous ranges of chunks (32 / TPP particles, one warp), so a block's
// gathers reuse its L1.  The sums over a particle's neighbours, the list rows and the
// thermostat's sum have the same order as in the separate kernels: results do not
// depend on which of them ran.
#pragma once
#include "k_force.cuh"
#include "team_core.cuh"

namespace gbmd {

//
// V = 2: one lane a particle does the sums of two (gather_mixed; TPP = 2, mixed), where the
// team has more than a turn of its warps' work at two lanes: half the warp instructions
// of the integration, whose FP64 pipe takes 16 cycles for each, and gathers of
// 32 neighbouring particles at once.  N = 64,000, 50 steps with readouts: 1,789 us by the
// step kernel and k_rebuild, 1,663 by the team.
template <int PREC, int TPP, int MT, int EVAL, int V = 1>
__global__ void __launch_bounds__(TEAM_T, 1) k_team(TeamArgs a) {
  constexpr int LP = TPP / V;   // lanes of a particle
  constexpr int T = TEAM_T, W = T / 32;
  extern __shared__ __align__(16) unsigned char team_smem_raw[];
  using Smem = TeamSmem<T, NL_SLOTS_TEAM>;
  Smem& sm = *reinterpret_cast<Smem*>(team_smem_raw);
  static_assert(sizeof(Smem) <= TEAM_SMEM, "team shared memory");
  __shared__ SplitTable tab;
  __shared__ unsigned slot[2 * TEAM_MAX_CLUSTER], word;
  __shared__ double nvt_sc;
  constexpr bool SMEM_TAB = PREC == GBMD_MIXED ? MT == 2 : MT != 0;
  __shared__ PairF tabf[SMEM_TAB ? MAXT2 : 1];
  __shared__ PairD tabd[SMEM_TAB && PREC == GBMD_FP64 ? MAXT2 : 1];
  Team tm;
  tm.cluster = a.cluster;
  tm.size = a.cluster ? a.cluster : (int)gridDim.x;
  tm.rank = a.cluster ? (int)(blockIdx.x % a.cluster) : (int)blockIdx.x;
  tm.sync = &a.ctl->team;
  int member = a.cluster ? (int)(blockIdx.x / a.cluster) : 0;
  if (a.share) {
    const int4 sh = a.share[blockIdx.x];
    member = sh.x;
    tm.rank = sh.y;
    tm.size = sh.z;
    tm.sync = a.sync + sh.w;
  }
  tm.gen = 0;
  tm.par = 0;
  tm.slot = slot;
  tm.word = &word;
  const SysDev& s = a.desc[a.list[member]];
  // The flags change only after the team's first barrier, so every block reads the same.
  const FlagWords fw = load_flag_words(s.flags);
  const longlong2 sl = load_flag_pair(&s.flags->step);        // (step, step_limit)
  const longlong2 lr = load_flag_pair(&s.flags->last_sort);   // (last_sort, n_rebuilds)
  const long long nsort0 = ((const volatile Flags*)s.flags)->n_sorts;
  if (!a.cluster) tm.gen = (unsigned)(*(const volatile unsigned long long*)&tm.sync->release >> 8);
  if (fw.error != 0 || (sl.y >= 0 && sl.x >= sl.y)) return;
  if (a.cluster) cooperative_groups::this_cluster().sync();   // every block runs: its shared
                                                              // memory may be written
  long long step = sl.x, last_sort = lr.x, rebuilds = lr.y, sorts = nsort0;
  int vfull = fw.v_full, error = 0;
  const int nt = s.ntypes, n = s.n;
  split_table(s, tab);
  if (SMEM_TAB)
    for (int k = threadIdx.x; k < nt * nt; k += blockDim.x) {
      tabf[k] = s.pf[k];
      if (PREC == GBMD_FP64) tabd[k] = s.pd[k];
    }
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = lane % LP;
  constexpr int PER = 32 / LP;   // particles of a chunk
  const int chunks = (n + PER - 1) / PER;
  const int c0 = (int)((long long)chunks * tm.rank / tm.size);
  const int c1 = (int)((long long)chunks * (tm.rank + 1) / tm.size);
  const bool nvt = s.nvt != 0;
  double xi = 0.0, eta = 0.0, sc = 1.0;
  if (nvt) {
    xi = s.nh[0];
    eta = s.nh[1];
    sc = s.nh[2];
  }
  for (int st = 0; st < a.nsteps; ++st) {
    if (sl.y >= 0 && step >= sl.y) break;
    bool need = false, bad = false;
    const int4* const qv = q_at(s, step);
    int4* const qn = q_at(s, step + 1);
    for (int c = c0 + w; c < c1; c += W) {
      const int g = c * PER + lane / LP;
      const bool valid = g < n;
      const int i = valid ? g : n - 1;
      const int nn = valid ? s.nn[i] : 0;
      if (valid && h == 0) prefetch_particle(s, i);
      double uu = 0.0;
      if constexpr (PREC == GBMD_MIXED) {
        const int4 qi = qv[i];
        float2 fx[V], fy[V], fz[V], e, wv[6];
        gather_mixed<LP, MT, EVAL, false, true, 2, V>(s, qv, qi, i, h, nn, tabf, fx, fy, fz, e, wv);
        auto total = [](const float2 (&f)[V]) {
          if constexpr (V == 2) return (f[0].x + f[0].y) + (f[1].x + f[1].y);
          else return group_sum<LP>(f[0].x + f[0].y);
        };
        const float Fx = total(fx), Fy = total(fy), Fz = total(fz);
        if (valid && h == 0) {
          const double f[3] = {widen_f32(Fx, bad), widen_f32(Fy, bad), widen_f32(Fz, bad)};
          if (nvt) {
            uu = nvt_close(s, i, f, vfull, sc);
            s.f32[i] = make_float4(Fx, Fy, Fz, 0.f);
          } else {
            bool moved = false;
            integrate_one<PREC>(s, i, qi.w, f, vfull, load_particle<true>(s, i), qn, nullptr, moved,
                                bad);
            need |= moved;
          }
        }
      } else {
        const longlong4_32a* const pv = p64_at(s, step);
        const longlong4_32a pi = pv[i];
        double fx, fy, fz, e, wv[6];
        gather_fp64<TPP, MT, EVAL, false, true>(s, pv, qv, pi, i, h, nn, tabf, tabd,
                                               sm.queue + threadIdx.x, T, fx, fy, fz, e, wv);
        fx = group_sum<TPP>(fx);
        fy = group_sum<TPP>(fy);
        fz = group_sum<TPP>(fz);
        if (valid && h == 0) {
          const double f[3] = {fx, fy, fz};
          if (nvt) {
            uu = nvt_close(s, i, f, vfull, sc);
            s.f64[i] = make_double4_32a(fx, fy, fz, 0.0);
          } else {
            bool moved = false;
            bad |= !isfinite(fx) || !isfinite(fy) || !isfinite(fz);
            integrate_one<PREC>(s, i, (int)pi.w, f, vfull,
                                load_particle<true>(s, i), qn, p64_at(s, step + 1), moved, bad);
            need |= moved;
          }
        }
      }
      if (nvt) {
        // V = 2: two of the sum's chunks, half a warp each, in the order of a warp of two
        // lanes a particle
        double part = uu;
        for (int o = V == 2 ? 8 : 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o, 32 / V);
        const int ch = V * c + lane / (32 / V);
        if (lane % (32 / V) == 0 && ch < s.nh_count) s.nh_part[s.nh_first + ch] = part;
      }
    }
    if (nvt) {
      // the thermostat between the halves: every block takes the same sum
      const unsigned v = tm.vote(bad ? VOTE_BAD : 0u);
      if (v & VOTE_LOST) { error = DEV_TEAM; break; }
      if (v & VOTE_BAD) { error = DEV_NONFINITE; break; }
      const double sum = nh_total<1>(s.nh_part + s.nh_first, s.nh_count, sm.sums);
      if (threadIdx.x == 0) nvt_sc = nh_update(s, sum, vfull, xi, eta);
      __syncthreads();
      sc = nvt_sc;
      // the opening half on this block's own particles
      const int p1 = min(n, c1 * PER);
      for (int i = c0 * PER + threadIdx.x; i < p1; i += T) {
        double f[3];
        if (PREC == GBMD_FP64) {
          const double4_32a F = s.f64[i];
          f[0] = F.x; f[1] = F.y; f[2] = F.z;
        } else {
          const float4 F = s.f32[i];
          f[0] = widen_f32(F.x, bad);
          f[1] = widen_f32(F.y, bad);
          f[2] = widen_f32(F.z, bad);
        }
        ParticleState p = load_particle<true>(s, i);
        for (int k = 0; k < 3; ++k) p.v[k] *= sc;
        bool moved = false;
        integrate_one<PREC>(s, i, s.type[i], f, 1, p, qn,
                            PREC == GBMD_FP64 ? p64_at(s, step + 1) : nullptr, moved, bad);
        need |= moved;
      }
    }
    const unsigned v = tm.vote((need ? VOTE_NEED : 0u) | (bad ? VOTE_BAD : 0u));
    if (v & VOTE_LOST) { error = DEV_TEAM; break; }
    if (v & VOTE_BAD) { error = DEV_NONFINITE; break; }
    ++step;
    vfull = 0;
    if (v & VOTE_NEED) {
      const int sp = s.sort_period;
      const bool sort = sp > 0 && step - last_sort >= sp;
      ++rebuilds;
      if (sort) {
        last_sort = step;
        ++sorts;
      }
      const unsigned r = team_rebuild<T, MT != 0>(s, tm, sm, tab, step, sort);
      if (r & VOTE_LOST) { error = DEV_TEAM; break; }
      if (r & VOTE_BAD) break;   // an overflowing row: the flags already say so
    }
  }
  if (tm.rank == 0 && threadIdx.x == 0) {
    volatile Flags* f = s.flags;
    f->step = step;
    f->v_full = vfull;
    f->rebuild_req = 0;
    f->do_rebuild = 0;
    f->do_sort = 0;
    f->active = error == 0;
    f->last_sort = last_sort;
    f->n_rebuilds = rebuilds;
    f->n_sorts = sorts;
    if (nvt) {
      s.nh[0] = xi;
      s.nh[1] = eta;
      s.nh[2] = sc;
    }
    if (error) atomicCAS(&s.flags->error, 0, error);
    atomicAdd(&s.flags->launches, 1ull);
    if (blockIdx.x == 0) atomicAdd(&a.ctl->launches, 1ull);
  }
}

// the team kernel for (precision, lanes per particle, table mode) with evaluator EVAL
template <int EVAL, int PREC, int TPP>
void* k_team_table(int mt) {
  if constexpr (PREC == GBMD_FP64 || EVAL != EVAL_LJ)
    return mt ? (void*)k_team<PREC, TPP, 2, EVAL> : (void*)k_team<PREC, TPP, 0, EVAL>;
  else
    return mt == 1   ? (void*)k_team<PREC, TPP, 1, EVAL>
           : mt == 2 ? (void*)k_team<PREC, TPP, 2, EVAL>
                     : (void*)k_team<PREC, TPP, 0, EVAL>;
}
template <int EVAL>
void* k_team_two_in_one(int mt) {
  if constexpr (EVAL != EVAL_LJ)
    return mt ? (void*)k_team<GBMD_MIXED, 2, 2, EVAL, 2> : (void*)k_team<GBMD_MIXED, 2, 0, EVAL, 2>;
  else
    return mt == 1   ? (void*)k_team<GBMD_MIXED, 2, 1, EVAL, 2>
           : mt == 2 ? (void*)k_team<GBMD_MIXED, 2, 2, EVAL, 2>
                     : (void*)k_team<GBMD_MIXED, 2, 0, EVAL, 2>;
}
template <int EVAL, int PREC>
void* k_team_tpp(int tpp, int mt, bool two_in_one) {
  if constexpr (PREC == GBMD_MIXED)
    if (tpp == 2 && two_in_one) return k_team_two_in_one<EVAL>(mt);
  return tpp == 1   ? k_team_table<EVAL, PREC, 1>(mt)
         : tpp == 2 ? k_team_table<EVAL, PREC, 2>(mt)
                    : k_team_table<EVAL, PREC, 4>(mt);
}

}  // namespace gbmd

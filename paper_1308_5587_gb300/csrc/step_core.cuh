// step_core.cuh -- the integration half of the fused step kernel (K5 + K6): the
// velocity-Verlet update of one particle once its force is known, and the end of
// the step (rebuild check, per-system decisions) done by the last block to finish.
//
// Velocity Verlet (Section 3.1 integrators; textbook form): with the stored velocity
// half a kick behind, step n of particle i is
//   v <- v + kick F_i(x^n),  kick = dt/m (closing half kick of step n-1 plus opening
//                            half kick of step n), or dt/(2m) right after create /
//                            set_state (v holds full-step velocities: Flags::v_full)
//   x <- x + dt v            (positions in box-fraction units x 2^32/L, so one FMA)
//   wrap into [-L/2, L/2), image += crossings, fixed-point shadow of x^{n+1}
// The shadows are double-buffered by step parity: the kernel of step n gathers
// neighbour positions from buffer n & 1 and writes x^{n+1} to the other one.
//
// FP64 runs at about 1/80 of the FP32 FMA rate on this part (measured: 1.6 against
// 128 FMAs per SM per clock), so the FP64 pipe only does the six FMAs of the kicks
// and drifts plus one add per axis: the FP32 force is widened to FP64 field by field
// on the integer pipe, and rint uses the 1.5 * 2^52 rounding constant.
#pragma once
#include "launch.cuh"

namespace gbmd {

// one thread: the system's flags and thermostat into its Snapshot
__device__ __forceinline__ void take_snapshot(const SysDev& s) {
  Snapshot* o = reinterpret_cast<Snapshot*>(s.thermo);
  const volatile long long* f = reinterpret_cast<const volatile long long*>(s.flags);
  long long* to = reinterpret_cast<long long*>(&o->flags);
  for (int k = 0; k < (int)(sizeof(Flags) / 8); ++k) to[k] = f[k];
  for (int k = 0; k < 3; ++k) o->nh[k] = s.nh[k];
}

// The row of particle i in a readout, at its tag, in the staging behind the Snapshot:
// force f, full-step velocity, position and image, as the bits of `what` ask
__device__ __forceinline__ void read_out(const SysDev& s, int i, const double (&f)[3], int vfull,
                                         int what) {
  const size_t n = (size_t)s.n, tg = (size_t)s.tag[i];
  double* const out = s.thermo + SNAPSHOT_BYTES / 8 + 3 * tg;
  int* const image = reinterpret_cast<int*>(s.thermo + SNAPSHOT_BYTES / 8 + 9 * n) + 3 * tg;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (what & READ_FORCE) out[a] = f[a];
    if (what & READ_VEL) {
      double v = s.v[a * n + i];
      if (!vfull) {
        v = fma(s.h, f[a], v);
        if (s.nvt) v *= s.nh[2];   // NVT: the closing thermostat scaling
      }
      out[3 * n + a] = v;
    }
    if (what & READ_POS) out[6 * n + a] = s.x[a * n + i] * (s.L[a] / 4294967296.0);
    if (what & READ_IMAGE) image[a] = s.img[a * n + i];
  }
}

// Eight values of every lane summed over the warp together: at distance 16 each half of
// the warp keeps four of them, at 8 two, at 4 one -- 9 FP64 additions where one shuffle
// tree after another takes 40.  Returns the sum of value lane / 4 to each four lanes.
__device__ __forceinline__ double warp_sum8(const double (&in)[8]) {
  const int lane = threadIdx.x & 31;
  double acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = in[c];
#pragma unroll
  for (int o = 16, keep = 4; o >= 4; o >>= 1, keep >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int c = 0; c < keep; ++c) {
      const double got = __shfl_xor_sync(0xffffffffu, up ? acc[c] : acc[c + keep], o);
      acc[c] = (up ? acc[c + keep] : acc[c]) + got;
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
  return acc[0];
}

// float -> double, exactly, on the integer pipe.  Zero and subnormal inputs (a
// force below 1.2e-38) give zero; inf / NaN set `bad`.
__device__ __forceinline__ double widen_f32(float f, bool& bad) {
  const unsigned u = __float_as_uint(f);
  const unsigned ex = (u >> 23) & 0xffu;
  bad |= ex == 0xffu;
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned long long mag = ((unsigned long long)(ex + 896u) << 52) |   // 1023 - 127
                                 ((unsigned long long)(u & 0x7fffffu) << 29);
  return __longlong_as_double((long long)(sign | (ex ? mag : 0ull)));
}

// rint(x) (ties to even) as an integer for |x| < 2^51: x + 1.5 * 2^52 lies in
// [2^52, 2^53), where the spacing of doubles is 1, so the sum is rounded to an
// integer and its bit pattern minus the constant's is that integer
__device__ __forceinline__ long long rint_ll(double x) {
  const double m = x + 6755399441055744.0;
  return __double_as_longlong(m) - 0x4338000000000000LL;
}

// the lines of the particle's state that the integration reads, requested into L2
// before the force loop (no registers held through the loop)
__device__ __forceinline__ void prefetch_particle(const SysDev& s, int i) {
  const int n = s.n;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(s.x + a * n + i));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(s.v + a * n + i));
  }
  asm volatile("prefetch.global.L2 [%0];" ::"l"(s.q_build + i));
}

// the particle's state the integration reads
struct ParticleState {
  double v[3], xq[3];
  int4 qb;   // shadow at the last list build
};
template <bool COH = false>   // COH: q_build may have been written by this kernel
__device__ __forceinline__ ParticleState load_particle(const SysDev& s, int i) {
  ParticleState p;
  const int n = s.n;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    p.v[a] = s.v[a * n + i];
    p.xq[a] = s.x[a * n + i];
  }
  p.qb = COH ? s.q_build[i] : __ldg(s.q_build + i);
  return p;
}

// one particle's kick, drift, wrap and new shadow; `need` = it moved more than
// r_buff/2 since the last list build
template <int PREC>
__device__ __forceinline__ void integrate_one(const SysDev& s, int i, int ty, const double f[3],
                                              int vfull, const ParticleState& p0,
                                              int4* __restrict__ q_next,
                                              longlong4_32a* __restrict__ p64_next, bool& need,
                                              bool& bad) {
  const int n = s.n;
  if (s.n_ghost > 0 && __ldg(s.tag + i) >= n - s.n_ghost) {
    // a ghost (a copy of a particle another domain owns) keeps the position set
    // before the step: no kick, drift or displacement check; the next shadow repeats
    // the current one
    const int4 qg = make_int4((int)rint_ll(p0.xq[0]), (int)rint_ll(p0.xq[1]),
                              (int)rint_ll(p0.xq[2]), ty);
    q_next[i] = qg;
    if (PREC == GBMD_FP64)
      p64_next[i] = fix_position(s, p0.xq[0], p0.xq[1], p0.xq[2], ty);
    return;
  }
  const double kick = vfull ? s.h : s.h + s.h;
  double v[3], xq[3];
  int q[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    v[a] = fma(kick, f[a], p0.v[a]);
    xq[a] = fma(s.dtq[a], v[a], p0.xq[a]);
    long long qq = rint_ll(xq[a]);
    const long long k = (qq + 0x80000000LL) >> 32;       // floor((xq + 2^31) / 2^32)
    if (k != 0) {
      if (k > 1 || k < -1 || !isfinite(xq[a])) bad = true;
      xq[a] -= (double)k * 4294967296.0;
      qq -= k << 32;
      s.img[a * n + i] += (int)k;
    }
    q[a] = (int)qq;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    s.v[a * n + i] = v[a];
    s.x[a * n + i] = xq[a];
  }
  q_next[i] = make_int4(q[0], q[1], q[2], ty);
  if (PREC == GBMD_FP64)
    p64_next[i] = fix_position(s, xq[0], xq[1], xq[2], ty);
  const float dx = (float)min_image_fixed(q[0], p0.qb.x) * s.fscale[0];
  const float dy = (float)min_image_fixed(q[1], p0.qb.y) * s.fscale[1];
  const float dz = (float)min_image_fixed(q[2], p0.qb.z) * s.fscale[2];
  need = dx * dx + dy * dy + dz * dz > s.rbuff_half2;
}

// NVT, first half at particle i once F_i(x^n) is known: the closing half kick and
// thermostat scaling of the previous step, u = (v + h F) exp(-xi dt/2) (just u = v
// right after create / set_state, when v holds full-step velocities); u is stored
// as the velocity and u.u returned for the kinetic energy.  The scale factor
// exp(-xi dt/2) is the one the previous step's opening half used (`sc`, nh[2]).
__device__ __forceinline__ double nvt_close(const SysDev& s, int i, const double f[3], int vfull,
                                            double sc) {
  const int n = s.n;
  double uu = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double u = s.v[a * n + i];
    if (!vfull) u = fma(s.h, f[a], u) * sc;
    s.v[a * n + i] = u;
    uu = fma(u, u, uu);
  }
  return uu;
}

// The sum of v.v over a system, in an order that depends on the lanes per particle alone
// and not on how the particles are spread over blocks or kernels: a warp's particles
// (32 / TPP consecutive ones, a chunk) by shuffles, the chunks' sums in NH_SLOTS strided
// slots, 32 slots at a time by shuffles, then those sums by shuffles.  In the team kernel
// every step waits for it: one barrier of the block (a tree in shared memory took eight;
// 50 NVT steps with readouts, N = 20,011: 1,746 us with it, 1,719 so).
constexpr int NH_SLOTS = 512, NH_SUMS = NH_SLOTS / 32;
__device__ __forceinline__ double nh_warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;   // lane 0
}
// Every thread of the block (whole warps) calls it; the sum is returned to all.  `sums`
// (shared) may be written again after the block's next barrier.  SIDE: slots that a thread
// sums side by side, four loads in flight for each (from L2: other blocks wrote them).  The
// team's 512 threads take one each; the tail of the step kernel's force half, often 128
// threads, four: one after another they were a chain of 20 such rounds at N = 160,000 (NVT,
// mixed: 90.8 us a step so, 86.4 side by side).
template <int SIDE>
__device__ __forceinline__ double nh_total(const double* part, int count, double* sums) {
  const int lane = threadIdx.x & 31, nt = (int)blockDim.x;
  // full rounds while the farthest slot of a thread has one (a block of more than a quarter
  // of the slots' threads has fewer slots side by side: the others read nothing); then a
  // slot has TAIL terms left at most
  constexpr int TAIL = SIDE == 1 ? 3 : 4;
  const int far = SIDE == 1 ? 0 : min((SIDE - 1) * nt, NH_SLOTS - 1);
  for (int v0 = threadIdx.x; v0 < NH_SLOTS; v0 += SIDE * nt) {   // the same for a warp's lanes
    double a[SIDE];
#pragma unroll
    for (int q = 0; q < SIDE; ++q) a[q] = 0.0;
    int k = v0;
    for (; k + far + 3 * NH_SLOTS < count; k += 4 * NH_SLOTS) {
      double p[SIDE][4];
#pragma unroll
      for (int q = 0; q < SIDE; ++q)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          p[q][u] = SIDE == 1 || v0 + q * nt < NH_SLOTS ? __ldcg(part + k + q * nt + u * NH_SLOTS) : 0.0;
#pragma unroll
      for (int q = 0; q < SIDE; ++q)
#pragma unroll
        for (int u = 0; u < 4; ++u) a[q] += p[q][u];
    }
    double p[SIDE][TAIL];
#pragma unroll
    for (int q = 0; q < SIDE; ++q)
#pragma unroll
      for (int u = 0; u < TAIL; ++u) {
        const int at = k + q * nt + u * NH_SLOTS;
        p[q][u] = (SIDE == 1 || v0 + q * nt < NH_SLOTS) && at < count ? __ldcg(part + at) : 0.0;
      }
#pragma unroll
    for (int q = 0; q < SIDE; ++q)
#pragma unroll
      for (int u = 0; u < TAIL; ++u) a[q] += p[q][u];
#pragma unroll
    for (int q = 0; q < SIDE; ++q) {
      const int v = v0 + q * nt;
      const double w = nh_warp_sum(a[q]);
      if (lane == 0 && v < NH_SLOTS) sums[v >> 5] = w;
    }
  }
  __syncthreads();
  double r = sums[lane & (NH_SUMS - 1)];
  for (int o = NH_SUMS / 2; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

// The thermostat (xi, eta) between two steps, from the sum of v.v of the closing
// velocities: the closing half of the previous step, then the opening half of this one,
// with G = (2K/(g kT) - 1)/tau^2 at their kinetic energy K:
//   eta += dt/2 xi;  xi += dt/2 G;     (skipped right after create / set_state)
//   xi += dt/2 G;    eta += dt/2 xi;   returns exp(-xi dt/2) for the opening scaling
__device__ __forceinline__ double nh_update(const SysDev& s, double sum, int vfull, double& xi,
                                            double& eta) {
  const double K = 0.5 * s.mass * sum;
  const double G = (2.0 * K / (s.gdof * s.kT) - 1.0) / (s.tau * s.tau);
  const double hdt = 0.5 * s.dt;
  if (!vfull) {
    eta += hdt * xi;
    xi += hdt * G;
  }
  xi += hdt * G;
  eta += hdt * xi;
  return exp(-hdt * xi);
}

// End of the NVT force half, every block: publish the warps' v.v sums (chunk `chunk` of
// the system for this warp, -1: none) and count the arrival; the last block of the system's
// own (nh_blocks of them) updates its thermostat.  (By the launch's last block for one
// system after another, us a step: 200 replicas of 500 1,118, so 231; 128 of 500 to 20,000
// 992 and 374; FP64 1,619 and 982.)
__device__ __forceinline__ void nvt_half_tail(const SysDev& s, double uu, int chunk) {
  const double part = nh_warp_sum(uu);
  if ((threadIdx.x & 31) == 0 && chunk >= 0) s.nh_part[s.nh_first + chunk] = part;
  __shared__ int last;
  __shared__ double sums[NH_SUMS];
  unsigned* const arrive = reinterpret_cast<unsigned*>(s.nh + 3);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(arrive, 1u) == (unsigned)s.nh_blocks - 1u);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) *arrive = 0u;
  // every block of the system has arrived: nothing writes its flags any more
  const FlagWords w = load_flag_words(s.flags);
  const longlong2 sl = load_flag_pair(&s.flags->step);
  if (!(w.error == 0 && (sl.y < 0 || sl.x < sl.y))) return;
  const double sum = nh_total<4>(s.nh_part + s.nh_first, s.nh_count, sums);
  if (threadIdx.x == 0) {
    double xi = s.nh[0], eta = s.nh[1];
    s.nh[2] = nh_update(s, sum, w.v_full, xi, eta);
    s.nh[0] = xi;
    s.nh[1] = eta;
  }
}

// End of the step, every block of the step's force launches: publish this block's
// rebuild request / error, count the arrival; the last of `total_blocks` arrivals
// makes each system's decisions for the next step (step counter, rebuild, re-sort)
// and sets the CUDA-graph conditional of the rebuild.  No block waits on another.
__device__ __forceinline__ void step_tail(const SysDev& s, const SysDev* __restrict__ sysv,
                                          GroupCtl* ctl, int nsys, int total_blocks,
                                          cudaGraphConditionalHandle cond, int use_cond,
                                          bool need, bool bad) {
  const int any_need = __syncthreads_or(need);
  const int any_bad = __syncthreads_or(bad);
  __shared__ int last;
  if (threadIdx.x == 0) {
    if (any_bad) atomicCAS(&s.flags->error, 0, (int)DEV_NONFINITE);
    if (any_need) atomicOr(&s.flags->rebuild_req, 1);
    __threadfence();
    last = (atomicAdd(&ctl->blocks_done, 1u) == (unsigned)total_blocks - 1u);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  int any = 0;
  for (int k = threadIdx.x; k < nsys; k += blockDim.x) {
    Flags* gf = sysv[k].flags;
    volatile Flags* g = gf;
    // every field the decision needs, in flight together; then the stores
    const FlagWords w = load_flag_words(gf);
    const longlong2 sl = load_flag_pair(&gf->step);        // (step, step_limit)
    const longlong2 lr = load_flag_pair(&gf->last_sort);   // (last_sort, n_rebuilds)
    const long long nsort = g->n_sorts;
    const int sp = sysv[k].sort_period;
    const bool act = w.error == 0 && (sl.y < 0 || sl.x < sl.y);
    // a domain with ghosts only records the request: its caller rebuilds every domain
    const bool ext = sysv[k].n_ghost > 0;
    if (act) {
      const long long st = sl.x + 1;
      const int req = w.rebuild_req;
      const int rb = ext ? 0 : req;
      const int srt = rb && sp > 0 && (st - lr.x >= sp);
      g->step = st;
      g->v_full = 0;
      g->rebuild_req = ext ? req : 0;
      g->do_rebuild = rb;
      if (rb) g->n_rebuilds = lr.y + 1;
      if (srt) {
        g->last_sort = st;
        g->n_sorts = nsort + 1;
      }
      g->do_sort = srt;
      g->active = 1;
      any |= rb;
    } else {
      g->active = 0;
      g->do_rebuild = 0;
      g->do_sort = 0;
    }
  }
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) {
    ctl->blocks_done = 0;
    ctl->any_rebuild = any;
    if (use_cond) cudaGraphSetConditional(cond, any ? 1u : 0u);
  }
}

}  // namespace gbmd

// fp64_math.cuh -- the FP64 pair force's arithmetic that is kept off the FP64 pipe.
//
// The FP64 pipe is the bound of the FP64 force path: it takes one warp instruction in
// 16 cycles of an SM (1.99 of 128 lanes a clock, measured), the time of some 30 integer
// instructions of each SM quarter.
#pragma once

namespace gbmd {

// ---- displacements and r^2 on the integer pipe ----
// A position is a 64-bit integer in units of 2^-fix_bits, chosen so that half the longest
// box edge is at most 2^61 units: an FP64 coordinate is held to 2^-62 of that edge or
// better, finer than its own last place for all but the smallest.  A displacement and
// the sum of its squares are then exact integers, and each is rounded to FP64 once.  On
// the FP64 pipe they are 6 of a pair's 17 instructions (three differences, r^2), each
// rounded.  20 steps with readouts, LJ 64,000: 3,970 -> 2,831 us; the paper's workload
// 4,182 -> 3,197.

// an integer below 2^62 with its highest word `hi` != 0, shifted left until its leading
// bit is bit 62 (`m`), as FP64: rounded to nearest at bit 10; `e` = (the biased exponent
// that bit 62 stands for) - 1, for the leading bit adds one to it
__device__ __forceinline__ double fix_pack(unsigned long long m, int e, unsigned sign) {
  const unsigned long long b = (m + 0x200ull) >> 10;
  return __hiloint2double((int)(((unsigned)(b >> 32) + ((unsigned)e << 20)) | sign), (int)(unsigned)b);
}

struct FixDiff {
  unsigned long long m;   // |d|
  unsigned sign;          // 0x80000000: d < 0
  __device__ __forceinline__ unsigned hi() const { return (unsigned)(m >> 32); }
  // the displacement through the other face: |d| -> L - |d|
  __device__ __forceinline__ void other_way(long long L) {
    m = (unsigned long long)L - m;
    sign ^= 0x80000000u;
  }
  // as FP64; sets `close` where |d| is below 2^32 units (2^-29 of half the edge, or 0) and
  // value_any is to be taken instead
  __device__ __forceinline__ double value(int fix_bits, bool& close) const {
    close |= hi() == 0u;
    const int sh = (__clz(hi()) - 1) & 31;
    return fix_pack(m << sh, 1022 + 62 - fix_bits - sh, sign);
  }
  __device__ __forceinline__ double value_any(int fix_bits) const {
    if (m == 0ull) return 0.0;
    const int lead = __clzll(m);   // 1 at least
    return fix_pack(m << (lead - 1), 1022 + 62 - fix_bits - (lead - 1), sign);
  }
};
__device__ __forceinline__ FixDiff fix_diff(long long a, long long b) {
  const long long d = a - b, s = d >> 63;
  return FixDiff{(unsigned long long)((d ^ s) - s), (unsigned)(d >> 32) & 0x80000000u};
}

// r^2 = m 2^(e - 1022 - 62): m with its leading bit at bit 62, or 0
struct FixR2 {
  unsigned long long m;
  int e;
  __device__ __forceinline__ double value() const { return m ? fix_pack(m, e, 0u) : 0.0; }
};

// |d|^2 of any size: all 128 bits of it
static __device__ __noinline__ FixR2 fix_r2_any(unsigned long long x, unsigned long long y,
                                                unsigned long long z, int fix_bits) {
  using u64 = unsigned long long;
  const unsigned __int128 r = (unsigned __int128)x * x + (unsigned __int128)y * y + (unsigned __int128)z * z;
  u64 s = (u64)(r >> 64);   // below 2^61
  u64 t = (u64)r;
  int e = 1022 + 126 - 2 * fix_bits;
  if (s == 0ull) {
    if (t == 0ull) return FixR2{0ull, 0};
    s = t;
    t = 0ull;
    e -= 64;
  }
  const int lead = __clzll(s);   // 0: one place too far left already
  const u64 m = lead == 0 ? s >> 1 : lead == 1 ? s : s << (lead - 1) | t >> (65 - lead);
  return FixR2{m, e - (lead - 1)};
}

// |d|^2 for components up to 2^61; sets `close` where it is below 2^96 units (r below 2^-13
// of half the longest edge) and fix_r2_any is to be taken instead
__device__ __forceinline__ FixR2 fix_r2(const FixDiff& x, const FixDiff& y, const FixDiff& z,
                                        int fix_bits, bool& close) {
  using u64 = unsigned long long;
  const unsigned xl = (unsigned)x.m, yl = (unsigned)y.m, zl = (unsigned)z.m;
  const unsigned xh = x.hi(), yh = y.hi(), zh = z.hi();   // <= 2^29
  const u64 high = (u64)xh * xh + (u64)yh * yh + (u64)zh * zh;      // x 2^64
  const u64 mid = (u64)xh * xl + (u64)yh * yl + (u64)zh * zl;       // x 2^33; below 2^63
  const u64 low = (u64)__umulhi(xl, xl) + __umulhi(yl, yl) + __umulhi(zl, zl);   // x 2^32
  // r^2 = (s 2^32 + t) 2^32, short of it by less than 3 2^32 (the low halves of the low
  // words' squares): 2^-62 of an r^2 of 2^96 and more
  const u64 a = (mid << 1) + low;
  const u64 s = high + (a >> 32);
  const unsigned t = (unsigned)a;
  close |= (unsigned)(s >> 32) == 0u;
  const int sh = (__clz((unsigned)(s >> 32)) - 1) & 31;   // 1 .. 30
  return FixR2{s << sh | t >> (32 - sh), 1022 + 126 - 2 * fix_bits - sh};
}

// ---- 1 / r^2 and its powers on the integer pipe ----
// With y = m 2^-62 in [1, 2): an FP32 approximation a0 of 1/y (24 bits) is refined by one
// step of the geometric series, e = 1 - y a0 exactly (below 2^-21 in magnitude, so the
// product's low 64 bits hold it): 1/y = a0 (1 + e + e^2 + ..), to 2^-59.  Its powers are
// the high parts of 64-bit products, to 2^-54; each used one is rounded to FP64 once.
// These replace the reciprocal's three FP64 instructions and three multiplications: a
// pair inside r_cut keeps 5 (the force factor's two, the three sums).  The results are
// within 0.61 ulp (compared with 128-bit arithmetic; the reciprocal below and two
// multiplications: up to 2).  20 steps with readouts, LJ 64,000: 2,831 -> 2,487 us; the
// paper's workload 3,197 -> 2,901.

// 2^62 / y
__device__ __forceinline__ unsigned long long fix_rcp(unsigned long long m) {
  using u64 = unsigned long long;
  const float y = __uint_as_float(((unsigned)(m >> 32) >> 7) + 0x3f000000u);   // 24 bits of y
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
  // a0 < 1 as 24 bits of 2^-24
  const unsigned a0 = (__float_as_uint(fminf(r, 0x1.fffffep-1f)) & 0x7fffffu) | 0x800000u;
  const long long p = (long long)((m >> 2) * a0);   // y a0 - 1 = -e, in 2^-84
  const int ph = (int)(p >> 32);                    // in 2^-52
  const long long t = ((long long)ph * ph >> 20) - p;   // e^2 + e
  const long long at = (t >> 24) * (int)a0;         // a0 (e + e^2) in 2^-84
  return ((u64)a0 << 38) + (u64)(at >> 22);
}
// a b 2^-62, less the low words' product
__device__ __forceinline__ unsigned long long fix_mul(unsigned long long a, unsigned long long b) {
  using u64 = unsigned long long;
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
  return ((u64)ah * bh << 2) + (((u64)ah * bl + (u64)al * bh) >> 30);
}
// f 2^-62 2^k as FP64 (f > 0 with a bit above bit 32)
__device__ __forceinline__ double fix_double(unsigned long long f, int k) {
  const int sh = __clz((unsigned)(f >> 32)) - 1;
  return fix_pack(f << sh, 1022 + k - sh, 0u);
}
// r^-2; r^-6 and r^-8.  r = 0: NaN
__device__ __forceinline__ double fix_inv2(const FixR2& q) {
  return q.m ? fix_double(fix_rcp(q.m), 1022 - q.e) : __longlong_as_double(0x7ff8000000000000ll);
}
__device__ __forceinline__ void fix_inv68(const FixR2& q, double& r6i, double& r8i) {
  const unsigned long long a = fix_rcp(q.m), a2 = fix_mul(a, a);
  const int k = 1022 - q.e;   // r^2 = y 2^-k
  r6i = fix_double(fix_mul(a2, a), 3 * k);
  r8i = fix_double(fix_mul(a2, a2), 4 * k);
  if (q.m == 0ull) r6i = r8i = __longlong_as_double(0x7ff8000000000000ll);
}

// ---- reciprocal on the FP64 pipe (the arithmetic probe's; the forces take the above) ----
// The correctly rounded reciprocal costs ~5.6 FMA slots.  Here the hardware approximation
// (rcp.approx.ftz.f64: relative error below 2^-19.9, measured over [0.25, 16)) is
// refined by one third-order step of the geometric series of 1/(1 - e):
//   a ~ 1/x,  e = 1 - x a,  1/x = a / (1 - e) = a (1 + e + e^2 + ...)  ->  a (1 + e + e^2)
// leaving a relative error of order e^3 < 2^-59 before rounding: within 1 ulp of
// the correctly rounded reciprocal (measured: 5,314 of 16.8 M inputs in [0.25, 16)
// differ by 1 ulp, none by more), for 3 FMAs plus the approximation (~3.3 slots).
// x must be positive and normal (r^2 > 0); at x = 0 the result is not finite and
// the step kernel's non-finite check reports it.
__device__ __forceinline__ double rcp_f64(double x) {
  double a;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(a) : "d"(x));
  const double e = fma(-x, a, 1.0);
  return fma(a, fma(e, e, e), a);
}

}  // namespace gbmd

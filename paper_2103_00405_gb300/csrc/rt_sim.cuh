// rt_sim.cuh -- per-event building blocks shared by the simulation kernels.
//
// Floating-point rules (so every mapping reproduces the same bits): each
// operation is one explicitly rounded binary64 op (__dadd_rn, __dsub_rn,
// __dmul_rn, __ddiv_rn; never contracted into an FMA).  Comparisons of values
// known to be non-negative (times, waiting times, propensities) are done on
// their bit patterns as signed 64-bit integers, which orders them exactly like
// the doubles and keeps the comparison off GB300's narrow FP64 pipe.
#pragma once
#include <cstdint>

#include "rt_filter.cuh"
#include "rt_internal.h"
#include "rt_rng.cuh"

namespace rt {

__device__ __forceinline__ int64_t dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double bitsd(int64_t b) { return __longlong_as_double(b); }
constexpr int64_t kInfBits = 0x7FF0000000000000ll;

// Exact binary64 value of 0 <= h < 2^53 built with integer instructions (the
// hardware int64 -> double conversion issues on the FP64 pipe); larger h rounds
// through the hardware conversion.
__device__ __forceinline__ double i64_to_f64(int64_t h) {
  if (h <= 0) return h == 0 ? 0.0 : __ll2double_rn(h);
  if (h >= (1ll << 53)) return __ll2double_rn(h);
  const int e = 63 - __clzll(h);  // position of the leading one, <= 52
  const uint64_t mant = (uint64_t)h << (52 - e);
  return __longlong_as_double((long long)((((uint64_t)(e + 1023)) << 52) | (mant & 0x000FFFFFFFFFFFFFull)));
}

// c * h rounded to nearest-even for a finite c >= 0 and an integer 0 <= h < 2^32,
// with integer instructions: the significand of c times h, normalised to 32 bits, is a
// 96-bit product whose leading bit is known up to one place.  Other operands use the
// FP64 pipe (identical result: h is exact in binary64).
__device__ __forceinline__ double mul_rn_pos_u32(double c, int64_t h) {
  if (h == 0) return 0.0;  // c is finite and >= 0
  const uint32_t ch = (uint32_t)__double2hiint(c), cl = (uint32_t)__double2loint(c);
  const uint32_t ec = ch >> 20;
  if ((uint64_t)h >> 32 || ec - 1u >= 2000u) return __dmul_rn(c, i64_to_f64(h));
  const int s = __clz((int)(uint32_t)h);
  const uint32_t hs = (uint32_t)h << s;
  const uint32_t mh = (ch << 11) | 0x80000000u | (cl >> 21), ml = cl << 11;  // significand of c, top bit set
  const uint64_t p0 = (uint64_t)ml * hs;
  uint64_t p = (uint64_t)mh * hs + (p0 >> 32);  // the product over 2^32, in [2^62, 2^64)
  uint32_t st = (uint32_t)p0;
  const bool top = (int64_t)p < 0;
  if (!top) {
    p = (p << 1) | (st >> 31);
    st <<= 1;
  }
  const uint32_t pl = (uint32_t)p;
  const bool up = (pl & 0x400u) != 0 && ((pl & 0xBFFu) | st) != 0;  // round bit, and odd or anything below it
  const uint64_t m = (p >> 11) + (up ? 1u : 0u);  // 53 bits; a carry out of them raises the exponent below
  return __longlong_as_double((long long)(((uint64_t)(ec + (top ? 31u : 30u) - (uint32_t)s) << 52) + m));
}

// 1 / x of a float by the special-function unit (at most 1 ulp off)
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// n / d rounded to nearest for n, d > 0, with integer instructions (a binary64 division keeps the
// FP64 pipe busy for about nine warp instructions of 16 cycles each, and each waits for the one
// before; this is some 60 integer instructions).  The significand quotient in [1, 2) is taken
// 30 and then 23 bits at a time, from a reciprocal good to 2^-29; the remainders are exact modulo
// 2^64, and the last one makes the 54-bit quotient the exact floor.  A quotient of two 53-bit
// significands is never half-way between two 53-bit numbers, so adding 1 and dropping the last bit
// rounds it to nearest.  Exponents far out (quotients that may not be normal) take the FP64 pipe.
// Measured with the product above: Lotka-Volterra ensemble 330 -> 265 ms, 64 Lotka-Volterra paths
// 359 -> 303 ms, 200-reaction network on warps 84.6 -> 74.8 ms.
__device__ __forceinline__ float mant_rcp(double d) {  // of d's significand, its first 24 bits
  const uint32_t D = __funnelshift_l((uint32_t)__double2loint(d), (uint32_t)__double2hiint(d), 3);
  return rcp_approx(__uint_as_float(0x3F800000u | (D & 0x7FFFFFu)));
}

__device__ __forceinline__ double div_rn_pos(double n, double d, float rcp_d) {  // rcp_d = mant_rcp(d)
  const uint32_t nh = (uint32_t)__double2hiint(n), nl = (uint32_t)__double2loint(n);
  const uint32_t dh = (uint32_t)__double2hiint(d), dl = (uint32_t)__double2loint(d);
  const uint32_t en = nh >> 20, ed = dh >> 20;
  if (!(en - 523u < 1000u && ed - 523u < 1000u)) return __ddiv_rn(n, d);
  const uint32_t mdh = (dh & 0xFFFFFu) | 0x100000u;
  const uint64_t mn = ((uint64_t)((nh & 0xFFFFFu) | 0x100000u) << 32) | nl, md = ((uint64_t)mdh << 32) | dl;
  const bool lt = mn < md;
  const uint64_t m = lt ? mn << 1 : mn;  // m / md in [1, 2)
  // r: 2^84 / md in [2^31, 2^32), from a float reciprocal biased below it (by more than the 2^-23 of
  // the dropped bits and the unit's error, at most 2^-20 in all) and one Newton step; off by -2..4
  const uint32_t D = __funnelshift_l(dl, mdh, 11);  // md 2^-21, top bit set
  const float y = fmaxf(rcp_d * 0.9999995f, 0.5f);
  uint32_t r = (__float_as_uint(y) << 8) | 0x80000000u;
  r += __umulhi(r, (0x80000000u - __umulhi(r, D)) << 1);
  const uint32_t q1 = __umulhi((uint32_t)(m >> 22), r) - 8u;    // below the quotient's 30 bits by 4 to 12
  const uint64_t r1 = (m << 30) - (uint64_t)q1 * md;            // in (0, 2^57)
  const uint32_t q2 = __umulhi((uint32_t)(r1 >> 25), r) >> 4;   // the next 23 bits, off by -1..1
  int64_t r2 = (int64_t)((r1 << 23) - (uint64_t)q2 * md);
  uint64_t q = ((uint64_t)q1 << 23) + q2;
  if (r2 < 0) {
    q -= 1;
    r2 += (int64_t)md;
  }
  if (r2 >= (int64_t)md) q += 1;
  return __longlong_as_double((long long)(((uint64_t)(en - ed + (lt ? 1021u : 1022u)) << 52) + ((q + 1) >> 1)));
}

__device__ __forceinline__ double div_rn_pos(double n, double d) { return div_rn_pos(n, d, mant_rcp(d)); }

// h_k(X) of Eq. 2 for a descriptor {s0, s1}, exact in int64, then a_k = c_k h_k (Eq. 1).
// IMUL: the product on integer instructions (faster where the FP64 pipe is the
// bottleneck) or on the FP64 pipe (the large-network scan, where the integer code
// in its loop costs more than it saves); both give the same bits.
template <bool IMUL = true, typename XAt>
__device__ __forceinline__ double propensity(int2 rd, double c, XAt x) {
  int64_t h;
  if (rd.x < 0) {
    h = 1;
  } else {
    const int64_t x0 = x(rd.x);
    if (rd.y == RD_UNI) h = x0;
    else if (rd.y == RD_DIMER) h = x0 * (x0 - 1) / 2;
    else h = x0 * (int64_t)x(rd.y);
  }
  return IMUL ? mul_rn_pos_u32(c, h) : __dmul_rn(c, i64_to_f64(h));
}

// Waiting time (P - T) / a of Eq. 25 for a > 0: 0 if no internal time is left.
__device__ __forceinline__ double waiting_time(double P, double T, double a) {
  const double rem = __dsub_rn(P, T);
  return dbits(rem) > 0 ? div_rn_pos(rem, a) : 0.0;
}

// Time-dependent rates c_k(t) = c_k (1 + beta_k t) (Sec. 6, Eq. 29): with A = c_k h_k(X)
// constant between events, the waiting time d solving A (d (1 + beta t) + beta d^2 / 2) = R
// for the remaining internal time R = P - T (the positive root, written without cancellation),
// and the integral of 1 + beta s over [t, t + d].  beta = 0 gives the constant-rate operations.
__device__ __forceinline__ double tdep_wait(double A, double beta, double R, double t) {
  if (!(dbits(R) > 0)) return 0.0;
  if (beta == 0.0) return __ddiv_rn(R, A);
  const double u = __dadd_rn(1.0, __dmul_rn(beta, t));
  const double b = __dmul_rn(A, u);
  const double e = __dmul_rn(__dmul_rn(__dmul_rn(2.0, A), beta), R);
  const double den = __dadd_rn(b, __dsqrt_rn(__dadd_rn(__dmul_rn(b, b), e)));
  return __ddiv_rn(__dmul_rn(2.0, R), den);
}

__device__ __forceinline__ double tdep_integral(double beta, double t, double d) {
  if (beta == 0.0) return d;
  const double u = __dadd_rn(1.0, __dmul_rn(beta, t));
  return __dadd_rn(__dmul_rn(d, u), __dmul_rn(__dmul_rn(__dmul_rn(beta, d), d), 0.5));
}

// The same from an already computed remainder rem = fl(P - T).
__device__ __forceinline__ double waiting_time_rem(double rem, double a) {
  return dbits(rem) > 0 ? div_rn_pos(rem, a) : 0.0;
}

// A float estimate of 1 / a, good to 2^-20 + 2^-23: +inf for a = 0 (the channel cannot fire), and 0
// for an a outside the estimates' range (its waiting-time estimate 0 sends the event to the exact path).
__device__ __forceinline__ float inv_estimate(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a);
  if (dbits(a) == 0) return __int_as_float(0x7F800000);
  return hi - (900u << 20) < (240u << 20) ? rcp_approx(__uint_as_float(hi * 8u - 0xC0000000u)) : 0.0f;
}

// An estimate of the quotient rem / a (rem > 0, a > 0) used only to pick which
// channel to compute exactly first; the exclusion test below is what is rigorous.
__device__ __forceinline__ float quot_estimate(double rem, double a) {
  return __fdividef(f32_upper(rem), f32_lower(a) + 1e-37f);
}

// True if the exact quotient rem / a is certainly > thr (rem > 0, a > 0).
__device__ __forceinline__ bool quot_exceeds(double rem, double a, float thr) {
  return f32_lower(rem) > __fmul_ru(thr, f32_upper(a));
}

// Float intervals of the waiting time (P - T) / a, kept per channel as {upper_P(P), inv_upper(a)}.
// A float >= P + 2^-125 (the term covers the floor of T's bound below); +inf from 2^127 on, where
// the interval becomes NaN and the channel is computed exactly.
__device__ __forceinline__ float upper_P(double P) {
  const uint32_t hi = (uint32_t)__double2hiint(P);
  return hi >= (1150u << 20) ? __int_as_float(0x7F800000) : __fadd_ru(f32_upper(P), 0x1p-125f);
}

// An upper bound of 1 / a, at most 2^-18 above it; +inf for a = 0 (the interval is at +inf); NaN where
// the float arithmetic could leave its range: never excluded, and ignored by the threshold.
__device__ __forceinline__ float inv_upper(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a);
  if (dbits(a) == 0) return __int_as_float(0x7F800000);
  return hi - (900u << 20) < (240u << 20) ? rcp_approx(__uint_as_float(hi * 8u - 0xC0000000u)) * 1.00000191f
                                          : __int_as_float(0x7FC00000);
}

// rem >= P - T >= rem - slack from the kept bound of P (the bound's excess is below 2^-19 P, that of
// T's float below 2^-20 T, and T exceeds P by a rounding at most).
__device__ __forceinline__ float rem_upper(float Pu, double T) {
  const uint32_t hi = max((uint32_t)__double2hiint(T), 897u << 20);
  return __fsub_ru(Pu, __uint_as_float(hi * 8u - 0xC0000000u));
}
__device__ __forceinline__ float rem_slack(float Pu) { return __fmaf_ru(Pu, 0x1p-18f, 0x1p-120f); }

// The upper end; lo is the lower end up to the factor that interval_threshold allows for.
__device__ __forceinline__ float wait_interval(float2 b, double T, float &lo) {
  const float rem = rem_upper(b.x, T);
  lo = __fmul_rd(__fsub_rd(rem, rem_slack(b.x)), b.y);
  return __fmul_ru(rem, b.y);
}

// A channel with lo above this has a waiting time above ub: the reciprocal's 2^-18 and the roundings
// of the exact operations are below 2^-17.
__device__ __forceinline__ float interval_threshold(float ub) { return __fmul_ru(fmaxf(ub, 0.0f), 1.00000763f); }

// Per-event trace: event ev of trajectory j fired channel mu at time t (recorded for
// the first trace_len events).
__device__ __forceinline__ void trace_event(const rt_outputs &o, int64_t j, int32_t ev, int mu, double t) {
  if (ev < o.trace_len) {
    if (o.trace_mu_dev) o.trace_mu_dev[j * o.trace_len + ev] = mu;
    if (o.trace_t_dev) o.trace_t_dev[j * o.trace_len + ev] = t;
  }
}

// The unused rest of trajectory j's trace, entries [ev, trace_len): -1 and 0, written
// by nthr cooperating threads (this one is number tid).
__device__ __forceinline__ void trace_tail(const rt_outputs &o, int64_t j, int32_t ev, int tid, int nthr) {
  for (int64_t e = (int64_t)ev + tid; e < o.trace_len; e += nthr) {
    if (o.trace_mu_dev) o.trace_mu_dev[j * o.trace_len + e] = -1;
    if (o.trace_t_dev) o.trace_t_dev[j * o.trace_len + e] = 0.0;
  }
}

// Register-array element r (runtime) by predicated selects, so arrays indexed with
// compile-time indices stay in registers.
template <int R, typename T>
__device__ __forceinline__ T pick(const T (&v)[R], int r) {
  T out = v[0];
#pragma unroll
  for (int i = 1; i < R; ++i) out = (i == r) ? v[i] : out;
  return out;
}

// lane of the lexicographic minimum of (w, k) over a warp, w >= 0 by its bits, k as an
// unsigned number (every lane calls it)
__device__ __forceinline__ int warp_argmin(long long w, int k) {
  const uint32_t hi = (uint32_t)(w >> 32), mh = __reduce_min_sync(0xFFFFFFFFu, hi);
  unsigned b = __ballot_sync(0xFFFFFFFFu, hi == mh);
  if (b & (b - 1)) {
    const uint32_t lo = hi == mh ? (uint32_t)w : 0xFFFFFFFFu, ml = __reduce_min_sync(0xFFFFFFFFu, lo);
    b = __ballot_sync(0xFFFFFFFFu, hi == mh && lo == ml);
    if (b & (b - 1)) {
      const bool in = hi == mh && lo == ml;
      const uint32_t mk = __reduce_min_sync(0xFFFFFFFFu, in ? (uint32_t)k : 0xFFFFFFFFu);
      b = __ballot_sync(0xFFFFFFFFu, in && (uint32_t)k == mk);
    }
  }
  return __ffs((int)b) - 1;
}

// a hint: bring the line holding p into L2 (no register result, never faults on a valid address)
__device__ __forceinline__ void prefetch_l2(const void *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

}  // namespace rt

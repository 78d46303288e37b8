// rt_rng.cuh -- device random draws for the random time algorithm.
//
// Eq. 24 of Liu & Wang (arXiv:2103.00405): each channel's internal-time
// increment is ln(1/r) with r uniform, i.e. Exp(1).  The uniform comes from
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11) keyed by the seed and
// indexed by (draw index >> 1, trajectory, channel, stream), so every channel is
// its own unit-rate Poisson process Y_k of Eq. 16 and any draw can be
// recomputed without state.
//
// The logarithm uses only integer instructions (GB300 issues 32-bit integer
// work at roughly fifty times its FP64 rate) and rounds once to binary64:
//   ln(M 2^E) = (E + q) ln2 + ln(m),  m = M / 2^q in [sqrt(1/2), sqrt(2)),
//   ln(m) = 2 atanh(s), s = (m - 1)/(m + 1), 2 atanh(s) = 2 s (1 + sum_i s^2i/(2i+1)),
// with s held in 64-bit fixed point (the quotient is the exact floor), the
// series to i = 12 by Horner's rule in Q64 (truncating products), ln2 as
// round(ln2 * 2^64), and a 128-bit fixed-point sum rounded to nearest-even.
// That evaluation (fx_ln) defines the value.  It costs some 300 instructions, and more in
// a warp whose lanes take its different branches, so a logarithm is first evaluated by
// tables (ln_tab, about 90 instructions, no branches), whose sum is known to lie within a
// few units of the 64th fractional bit of fx_ln's: unless a rounding boundary lies that
// close, both round to the same binary64.  Otherwise (0.5 % of the Exp(1) draws) fx_ln runs.
// Measured against fx_ln alone: 250001 Lotka-Volterra trajectories to t = 1 438 -> 330 ms, the
// likelihood and gradient of a 64-reaction network (65536 trajectories) 459 -> 370 ms, 64
// Lotka-Volterra paths to t = 5 447 -> 359 ms (there the draw is on each event's critical path).
#pragma once
#include <cstdint>

#include "rt_lntab.cuh"

namespace rt {

typedef unsigned __int128 u128;

// ---------------------------------------------------------------------------
// Philox4x32-10
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// 64 random bits of draw `n` of channel k in trajectory g.
__device__ __forceinline__ uint64_t draw_bits(uint64_t seed, uint64_t g, uint32_t k, uint32_t n, uint32_t stream) {
  const uint4 o = philox4x32_10(make_uint4(n >> 1, (uint32_t)g, k, stream), (uint32_t)seed, (uint32_t)(seed >> 32));
  const uint32_t w0 = (n & 1u) ? o.z : o.x;
  const uint32_t w1 = (n & 1u) ? o.w : o.y;
  return ((uint64_t)w1 << 32) | w0;
}

// ---------------------------------------------------------------------------
// 128-bit helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ int clz128(u128 v) {
  const uint64_t hi = (uint64_t)(v >> 64), lo = (uint64_t)v;
  return hi ? __clzll(hi) : 64 + __clzll(lo);
}

// Nearest binary64 to V * 2^scale (V > 0), ties to even; result known to be normal.
__device__ __forceinline__ double round_to_f64(u128 V, int scale) {
  const int p = 127 - clz128(V);
  uint64_t mant;
  int e = p;
  if (p <= 52) {
    mant = (uint64_t)V << (52 - p);
  } else {
    const int sh = p - 52;
    uint64_t q = (uint64_t)(V >> sh);
    const u128 rem = V & (((u128)1 << sh) - 1);
    const u128 half = (u128)1 << (sh - 1);
    q += (rem > half || (rem == half && (q & 1))) ? 1 : 0;
    if (q >> 53) {
      q >>= 1;
      e += 1;
    }
    mant = q;
  }
  const uint64_t bits = ((uint64_t)(e + scale + 1023) << 52) | (mant & 0x000FFFFFFFFFFFFFull);
  return __longlong_as_double((long long)bits);
}

// floor(n * 2^63 / d) for n, d in [2^63, 2^64).  x = 2^64 + v approximates
// 2^128 / d from below: a float reciprocal of d rounded up, itself rounded toward
// zero, then two Newton steps x += x (2^128 - d x) / 2^128 with truncated
// products.  Newton's reciprocal iteration started below the root stays below it
// and increases, so v never wraps; the quotient estimate is then at most a few
// units low and is made exact by comparing the remainder with d.
__device__ __forceinline__ uint64_t quot_q63(uint64_t n, uint64_t d) {
  const float r = __frcp_rz((float)((uint32_t)(d >> 40) + 1u));  // <= 2^40 / d, in [2^-24, 2^-23)
  const uint64_t R = __float2ull_rz(r * 0x1p62f);                 // in [2^38, 2^39)
  uint64_t v = (R - (1ull << 38)) << 26;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const u128 dx = ((u128)d << 64) + (u128)d * v;
    const uint64_t ehi = (uint64_t)((((u128)0) - dx) >> 64);  // (2^128 - d x) / 2^64 >= 0
    v += ehi + __umul64hi(v, ehi);
  }
  uint64_t q = (uint64_t)(((u128)n + __umul64hi(n, v)) >> 1);
  u128 rem = ((u128)n << 63) - (u128)q * d;  // >= 0: q is not above the quotient
#pragma unroll 1
  for (int i = 0; i < 8 && rem >= (u128)d; ++i) {
    q += 1;
    rem -= d;
  }
  return q;
}

// ln(M * 2^E) for integer 1 <= M < 2^53.
__device__ __forceinline__ double fx_ln(uint64_t M, int E) {
  int q = 63 - __clzll(M);
  if ((u128)M * M >= ((u128)1 << (2 * q + 1))) q += 1;
  const int K = E + q;
  const uint64_t P = 1ull << q;
  const uint64_t n = M >= P ? M - P : P - M;
  const uint64_t d = M + P;
  if (n == 0) {
    if (K == 0) return 0.0;
    const u128 A = (u128)(uint64_t)(K > 0 ? K : -K) * 0xB17217F7D1CF79ACull;
    const double r = round_to_f64(A, -64);
    return K > 0 ? r : -r;
  }
  const int a = __clzll(n), b = __clzll(d);
  const uint64_t Q = quot_q63(n << a, d << b);  // |s| = Q 2^(b - a - 63)
  const int sh = a - b - 1;                     // >= 1
  const uint64_t s64 = sh >= 64 ? 0ull : (Q >> sh);
  const uint64_t z = __umul64hi(s64, s64);
  // sum_{i=1..12} z^i/(2i+1) in Q64; constants are floor(2^64 / (2i+1))
  uint64_t R = 0xFFFFFFFFFFFFFFFFull / 25u;
  R = 0xFFFFFFFFFFFFFFFFull / 23u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 21u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 19u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 17u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 15u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 13u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 11u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 9u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 7u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 5u + __umul64hi(z, R);
  R = 0xFFFFFFFFFFFFFFFFull / 3u + __umul64hi(z, R);
  const uint64_t F = __umul64hi(z, R);
  const u128 Lm = (u128)Q + __umul64hi(Q, F);  // |ln m| = Lm 2^(b - a - 62)
  const bool pos = M > P;                      // sign of ln m
  if (K == 0) {
    const double r = round_to_f64(Lm, b - a - 62);
    return pos ? r : -r;
  }
  const int rs = a - b - 2;  // |ln m| in Q64 = Lm >> rs
  const u128 LQ = rs >= 128 ? (u128)0 : (Lm >> rs);
  const u128 A = (u128)(uint64_t)(K > 0 ? K : -K) * 0xB17217F7D1CF79ACull;
  if (K > 0) return round_to_f64(pos ? A + LQ : A - LQ, -64);
  return -round_to_f64(pos ? A - LQ : A + LQ, -64);
}

// ln by tables.  x = f 2^53 (53 bits, top bit set).
//   NEG false: the bits of V = k ln2 - ln f, k >= 0 (minus the logarithm of f 2^-k)
//   NEG true:  the bits of V = k ln2 + ln f, k >= 2 (the logarithm of f 2^k)
// Returns false where V and fx_ln's sum might round differently (then *bits is meaningless).
//
// f r = 1 - z from kLn1 (exact: z in Q68), (1 - z)(1 + t) = 1 - z' from kLn2 (z' < 2^-11.9,
// Q68, error < 1 unit), so -ln f = ln r + ln(1 + t) + z' + z'^2/2 + z'^3 (1/3 + z'/4 + z'^2/5).
// The truncations sum to less than 2^-65, all to one side, plus 2^-69 of the tables'
// rounding.  ln 2 enters with the constant of fx_ln, so it adds no difference.  fx_ln's sum
// lies below the true value of |ln m| by at most (units of 2^-64) 1 + 0.53 for the floors of
// Q and of F's series and 1 for the product: 2.54; with K = 0, where it keeps the scale of
// |ln m| itself, by at most 2.8 units of Lm, whose leading bit is bit 62 or above: 5.6 units
// of the 64-bit normalised N below.  `below` and `above` are these bounds in units of N.
template <bool NEG>
__device__ __forceinline__ bool ln_tab(uint64_t x, int k, uint64_t &bits) {
  const Ln1Entry e1 = ln1_entry((uint32_t)(x >> 46) - 64u);
  const uint64_t z = 0ull - x * (uint64_t)e1.r;  // Q68, < 2^62.1
  const Ln2Entry e2 = ln2_entry((uint32_t)(z >> 56));
  const uint32_t zh = (uint32_t)(z >> 32), zl = (uint32_t)z;
  const uint64_t zp = z + ((uint64_t)zh * e2.t + __umulhi(zl, e2.t)) - ((uint64_t)(e2.t << 4) << 32);  // z', Q68
  const uint32_t yh = (uint32_t)(zp >> 25), yl = (uint32_t)zp << 7;                   // z' in Q75
  const uint64_t sq = (uint64_t)yh * yh + ((uint64_t)__umulhi(yh, yl) << 1);          // z'^2, Q86
  uint32_t u = 0x40000000u + (__umulhi(yh, 0x33333333u) >> 11);                       // 1/4 + z'/5, Q32
  u = 0x55555555u + (__umulhi(yh, u) >> 11);                                          // 1/3 + z' u
  const uint32_t g = (uint32_t)(((uint64_t)yh * u) >> 30);                            // z' u, Q45
  const uint64_t S = zp + (sq >> 19) + ((uint64_t)__umulhi((uint32_t)(sq >> 32), g) << 1);  // -ln(1 - z'), Q68
  const uint64_t W = e1.L + e2.L;  // two's complement Q64, |W| < 1/2
  const uint32_t half = e1.info & 1u;
  const uint32_t kk = NEG ? (uint32_t)k - half : (uint32_t)k + half;
  const uint64_t c0 = (uint64_t)kk * 0xD1CF79ACu;
  const uint64_t c1 = (uint64_t)kk * 0xB17217F7u + (c0 >> 32);
  const uint64_t kl = (c1 << 32) | (uint32_t)c0;  // kk ln2: fraction, and the integer part c1 >> 32
  uint32_t w2 = (uint32_t)(c1 >> 32), w1, w0, gd;
  if (!NEG) {
    const uint64_t a = kl + W;
    w2 += (uint32_t)((int32_t)(uint32_t)(W >> 32) >> 31) + (a < kl ? 1u : 0u);
    const uint64_t b = a + (S >> 4);
    w2 += b < a ? 1u : 0u;
    w1 = (uint32_t)(b >> 32);
    w0 = (uint32_t)b;
    gd = (uint32_t)S << 28;
  } else {
    const uint64_t q = W + (S >> 4);  // |q| < 1/2
    const uint64_t a = kl - q;
    w2 -= (uint32_t)((int32_t)(uint32_t)(q >> 32) >> 31) + (kl < q ? 1u : 0u);
    w1 = (uint32_t)(a >> 32);
    w0 = (uint32_t)a;
    gd = 0u;
  }
  const bool frac = w2 == 0u;  // V < 1
  int e = 31;
  if (frac) {
    w2 = w1;
    w1 = w0;
    w0 = gd;
    e = -1;
  }
  const int s = __clz((int)w2);
  const uint32_t nh = __funnelshift_l(w1, w2, s), nl = __funnelshift_l(w0, w1, s);  // N, top bit set
  const uint32_t unit = frac ? 1u << min(s, 12) : 1u;  // 2^-64 in units of N, rounded up to 1
  const uint32_t base = kk == 0u ? 6u : 3u * unit;
  const uint32_t lo = (e1.info & (NEG ? 4u : 2u)) ? base : 0u, hi = (e1.info & (NEG ? 2u : 4u)) ? base : 0u;
  const uint32_t below = lo + (NEG ? 3u : 1u + (unit >> 4)), above = hi + (NEG ? 3u : 1u + (unit >> 1));
  const uint32_t pos = (nl + 0x400u - below) & 0x7FFu;  // distance of N - below from the rounding boundary under it
  const uint64_t m = (((uint64_t)nh << 21) | (nl >> 11)) + ((nl >> 10) & 1u);
  bits = ((uint64_t)(uint32_t)(e - s + 1022) << 52) + m;
  return pos + below + above <= 0x7FFu;
}

// ln(x) of a positive finite binary64.
__device__ __forceinline__ double rt_ln(double x) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
  const int ef = (int)((bits >> 52) & 0x7FF);
  const uint64_t frac = bits & 0x000FFFFFFFFFFFFFull;
  uint64_t r;
  if (ef >= 1024 && ln_tab<true>(frac | (1ull << 52), ef - 1022, r)) return __longlong_as_double((long long)r);
  return ef == 0 ? fx_ln(frac, -1074) : fx_ln(frac | (1ull << 52), ef - 1075);
}

// The odd integer x with u = x 2^-53 for 64 random bits.
__device__ __forceinline__ uint64_t bits_to_x(uint64_t bits) { return ((bits >> 12) << 1) | 1ull; }

// Exp(1) increment ln(1/u) (Eq. 24).
__device__ __forceinline__ double exp1_from_bits(uint64_t bits) {
  const uint64_t x = bits_to_x(bits);
  const int lz = __clzll((long long)x) - 11;
  uint64_t r;
  if (ln_tab<false>(x << lz, lz, r)) return __longlong_as_double((long long)r);
  return -fx_ln(x, -53);
}

__device__ __forceinline__ double exp1_draw(uint64_t seed, uint64_t g, uint32_t k, uint32_t n, uint32_t stream) {
  return exp1_from_bits(draw_bits(seed, g, k, n, stream));
}

}  // namespace rt

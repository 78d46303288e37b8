// rt_traj_warp.cuh -- trajectories in warp segments: G lanes per trajectory, 32 / G
// trajectories per warp (channel k in sub-lane k % G, slot k / G).
//
// The NRRTA loop of Table 2 (Liu & Wang, arXiv:2103.00405), each trajectory's channels
// spread over the G lanes of its segment (Eq. 17-27).  Only the internal times T_k live in
// registers; P_k, a_k, the increment drawn ahead for the channel's next firing, its firing
// count and two floats (an upper bound of P_k, and of 1 / a_k) are in shared memory, so that
// with eight channels per lane five or six blocks of four warps fit on an SM, and so
// that the propensities an event changed can be recomputed by any lane of the segment: its
// list of dependent channels is dealt out to the lanes one each.
//
// GB300 issues a binary64 warp instruction every 16 cycles per SM and its result takes 64;
// the advance T_k += a_k dt of every channel at every event (two of them) is the work the
// method fixes.  Everything else stays off that pipe or is shared by the trajectories of the
// warp: per channel a float interval of the waiting time (Pu - T) / a decides whether it can
// be the smallest -- a segment minimum of the upper ends is the threshold -- and only channels
// that can are computed exactly (integer division, each lane its next such channel per pass);
// usually there is one per segment and a vote finds it.  When the increment that a firing needs is
// not there, every lane draws one that its channels lack, the owner of the fired channel that one
// (drawing all that are lacking each time, and one per channel at the start, made a run without
// events, 100000 trajectories of 256 reactions, 4.9 ms instead of 1.9, and 65536 trajectories of 64
// reactions with likelihood and gradient 177 instead of 169 ms), and with the likelihood ln a_mu is taken G events at a time, one event per lane.  Trajectories of one
// warp advance event by event together; a finished one leaves its lanes idle until the others
// finish.  The network arrays may live in shared or global memory (generic pointers).
//
// TD: time-dependent rates c_k(t) = c_k (1 + beta_k t) (Sec. 6, Eq. 29): T_k advances by its
// channel's integral and the interval is that of the integral's root, in floats.
#pragma once
#include <climits>

#include "rt_sim.cuh"

namespace rt {

struct WarpNet {
  int M, N;
  const int2 *rd;
  const double *c;
  const int *vp;
  const int2 *vl;
  const int *dptr;     // per reaction the channels its firing touches: dlist[dptr[k]..dptr[k+1])
  const int *dlist;
  const double *beta;  // TD: rate slopes
};

// Shared memory of one trajectory: P, a, E (binary64), the float pair, n, X; arrays padded to a
// multiple of the segment width, the whole to an odd multiple of 64 bytes so that the four segments
// of G = 8 start in different banks.
__host__ __device__ inline int warp_pad(int M, int G) { return (M + G - 1) / G * G; }
__host__ __device__ inline size_t warp_seg_bytes(int M, int N, int G) {
  const size_t b = (size_t)warp_pad(M, G) * 36 + (size_t)N * 4;
  return (b + 63) / 128 * 128 + 64;
}

struct WarpSeg {
  double *P, *a, *E;
  float2 *b;
  int *n, *X;
};

__device__ __forceinline__ WarpSeg carve_warp_seg(unsigned char *base, int Mp) {
  WarpSeg s;
  s.P = (double *)base;
  s.a = s.P + Mp;
  s.E = s.a + Mp;
  s.b = (float2 *)(s.E + Mp);
  s.n = (int *)(s.b + Mp);
  s.X = s.n + Mp;
  return s;
}

// The float kept with a propensity: inv_upper, or for TD a lower bound of a (+inf for a = 0, NaN
// outside the range of its float arithmetic).
template <bool TD>
__device__ __forceinline__ float warp_rate_bound(double a) {
  if (!TD) return inv_upper(a);
  const uint32_t hi = (uint32_t)__double2hiint(a);
  if (dbits(a) == 0) return __int_as_float(0x7F800000);
  return hi - (983u << 20) < (80u << 20) ? __uint_as_float(hi * 8u - 0xC0000000u) : __int_as_float(0x7FC00000);
}
// The log-likelihood's sum_k T_k in k order for every segment of the warp (all lanes call it;
// segments past n_traj pass live = false).
template <int R, int G>
__device__ __forceinline__ double warp_sum_T_in_order(const double (&T)[R], int M, bool live) {
  const int lane = threadIdx.x & 31, base = (lane / G) * G;
  double sT = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r)
    for (int l = 0; l < G; ++l) {
      const double v = __shfl_sync(0xFFFFFFFFu, T[r], base + l);
      if (live && l + G * r < M) sT = __dadd_rn(sT, v);
    }
  return sT;
}

// Trajectories j0 .. j0 + 32/G - 1 (those < n_traj) in the segments of one warp.  base: the
// warp's shared memory, 32/G times warp_seg_bytes; mom: block moment table (or null).
template <int R, int G, bool LL, bool TD>
__device__ __forceinline__ void warp_trajectories(const RunArgs &A, const WarpNet &net, unsigned char *base_mem,
                                                  unsigned long long *mom, const int64_t j0, const int tend_finite) {
  static_assert(G == 8 || G == 16 || G == 32, "segment width");
  constexpr unsigned FULL = 0xFFFFFFFFu;
  const float INF = __int_as_float(0x7F800000);
  const int lane = threadIdx.x & 31, seg = lane / G, sl = lane % G, base = seg * G;
  const unsigned segmask = G == 32 ? FULL : (((1u << (G & 31)) - 1u) << base);
  const int M = net.M, N = net.N, Mp = warp_pad(M, G);
  const int64_t j = j0 + seg;
  const bool live = j < A.n_traj;
  const WarpSeg S = carve_warp_seg(base_mem + (size_t)seg * warp_seg_bytes(M, N, G), Mp);
  int *X = S.X;
  const uint64_t g = (uint64_t)(A.traj_offset + j);
  const int32_t *x0 = A.x0 + (A.per_traj_x0 ? j * (int64_t)N : 0);
  bool badl = false;
  if (live)
    for (int s = sl; s < N; s += G) {
      const int v = x0[s];
      X[s] = v;
      badl |= v < 0;
    }
  const bool bad = (__ballot_sync(FULL, badl) & segmask) != 0;
  __syncwarp();
  auto xat = [&](int s) { return X[s]; };
  const int64_t GN = A.G * N;

  auto record = [&](int64_t gidx, bool known) {  // the segment's lanes
    if (A.out.grid_dev) {
      int32_t *gp = A.out.grid_dev + (j * A.G + gidx) * N;
      for (int s = sl; s < N; s += G) gp[s] = known ? X[s] : -1;
    }
    if (!known || !A.out.grid_sum_dev) return;
    for (int s = sl; s < N; s += G) {
      const long long x = X[s];
      if (mom) {
        atomicAdd(mom + gidx * N + s, (unsigned long long)x);
        atomicAdd(mom + GN + gidx * N + s, (unsigned long long)(x * x));
      } else {
        atomicAdd((unsigned long long *)(A.out.grid_sum_dev + gidx * N + s), (unsigned long long)x);
        if (A.out.grid_sumsq_dev)
          atomicAdd((unsigned long long *)(A.out.grid_sumsq_dev + gidx * N + s), (unsigned long long)(x * x));
      }
    }
    if (sl == 0) {
      if (mom) atomicAdd(mom + 2 * GN + gidx, 1ull);
      else if (A.out.grid_count_dev) atomicAdd((unsigned long long *)(A.out.grid_count_dev + gidx), 1ull);
    }
  };

  double T[R];
  bool run = live && !bad;  // segment-uniform: this trajectory still fires events
  uint32_t stale = 0;       // bit r: the increment of slot r's channel is used up or not drawn yet (its E is -1)
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int k = sl + G * r;
    T[r] = 0.0;
    if (G * r < M) {
      double P = 1.0, a = 0.0;  // past M: a = 0 and an interval at +inf
      if (run && k < M) {
        P = exp1_draw(A.seed, g, (uint32_t)k, 0u, A.stream_id);
        a = propensity(net.rd[k], net.c[k], xat);
        stale |= 1u << r;
      }
      S.P[k] = P;
      S.E[k] = -1.0;
      S.a[k] = a;
      S.n[k] = 0;
      S.b[k] = make_float2(upper_P(P), warp_rate_bound<TD>(a));
    }
  }
  int status = bad ? RT_TRAJ_BAD_X0 : RT_TRAJ_TEND;
  double t = 0.0, ll = 0.0, dprev = 0.0, tprev = 0.0;
  double ring = 0.0;  // with the likelihood: a_mu of event (ev & ~(G-1)) + sl of this trajectory
  int db = 0, de = 0;  // the last firing's dependent channels dlist[db..de)
  int32_t ev = 0;
  int64_t gi = 0;
  double next_g = 0.0;
  const int64_t tend_bits = dbits(A.t_end);

  // ll += ln a_mu of the cnt buffered events of each segment, in event order (the segment's
  // lanes take the logarithms together); cnt is segment-uniform, 0..G
  auto flush_ring = [&](int cnt) {
    double L = 0.0;
    if (sl < cnt) L = rt_ln(ring);
    for (int i = 0; i < G; ++i) {
      const double v = __shfl_sync(FULL, L, base + i);
      if (sl == 0 && i < cnt) ll = __dadd_rn(ll, v);
    }
  };
  __syncwarp();

  while (__any_sync(FULL, run)) {
    // ---- internal times advance with the pre-event propensities (Eq. 17)
    if (run && dbits(dprev) != 0) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (G * r < M) {
          const int k = sl + G * r;
          if (TD) {
            if (k < M) T[r] = __dadd_rn(T[r], __dmul_rn(S.a[k], tdep_integral(net.beta[k], tprev, dprev)));
          } else {
            T[r] = __dadd_rn(T[r], __dmul_rn(S.a[k], dprev));  // a = 0 in the padding
          }
        }
    }
    __syncwarp();
    // ---- propensities the last firing changed (Eq. 1-2), dealt out to the segment's lanes
    for (int i = db + sl; __any_sync(FULL, i < de); i += G)
      if (i < de) {
        const int k = net.dlist[i];
        const double v = propensity(net.rd[k], net.c[k], xat);
        S.a[k] = v;
        S.b[k].y = warp_rate_bound<TD>(v);
      }
    __syncwarp();
    // ---- float intervals of the waiting times; the segment minimum of the upper ends
    float ub = INF;
    float lo[R];
    const float NANF = __int_as_float(0x7FC00000);
    const float tf = TD ? (dbits(t) < dbits(1e18) ? f32_lower(t) : NANF) : 0.0f;
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (G * r < M) {
        const int k = sl + G * r;
        const float2 q = S.b[k];
        if (TD) {
          const float rem = rem_upper(q.x, T[r]);
          const float bf = k < M ? f32_lower(net.beta[k]) : 0.0f;
          const float bb = q.y * __fmaf_rn(bf, tf, 1.0f);
          const float d2 = bb * bb + 2.0f * q.y * bf * fmaxf(rem, 0.0f);
          float y = 2.0f * rcp_approx(bb + sqrt_approx(d2)) * 1.0000077f;  // waiting time over remaining internal time
          y = d2 < 1e37f && bf < 1e18f && rem < 1e18f ? y : NANF;  // ranges in which the errors are bounded
          y = q.y == INF ? INF : y;
          ub = fminf(ub, __fmul_ru(rem, y));  // a NaN is ignored
          lo[r] = __fmul_rd(__fsub_rd(rem, rem_slack(q.x)), y);
        } else {
          ub = fminf(ub, wait_interval(q, T[r], lo[r]));
        }
      }
    if (!run) ub = INF;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) ub = fminf(ub, __shfl_xor_sync(FULL, ub, o));
    // ---- exact waiting times (Eq. 25) of the channels whose interval reaches below the threshold
    // (widened for the error of y): each lane its next such channel per pass
    const float thr = TD ? __fmul_ru(fmaxf(ub, 0.0f), 1.00006104f) : interval_threshold(ub);
    uint32_t need = 0;
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (G * r < M && run && !(lo[r] > thr)) need |= 1u << r;
    const unsigned nb = __ballot_sync(FULL, need != 0) & segmask;
    long long bw = kInfBits;
    int bk = INT_MAX;
    while (__any_sync(FULL, need != 0)) {
      if (need) {
        const int r = __ffs((int)need) - 1;
        const int k = sl + G * r;
        const double ak = S.a[k], rem = __dsub_rn(S.P[k], pick<R>(T, r));
        need &= need - 1;
        if (dbits(ak) != 0) {
          const long long wb = dbits(TD ? tdep_wait(ak, net.beta[k], rem, t) : waiting_time_rem(rem, ak));
          if (wb < bw || (wb == bw && k < bk && wb != kInfBits)) {
            bw = wb;
            bk = k;
          }
        }
      }
    }
    // the segment's exact argmin, smallest index on ties (Eq. 26); a lone candidate needs no reduction
    if (__any_sync(FULL, (nb & (nb - 1)) != 0)) {
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        const long long w2 = __shfl_xor_sync(FULL, bw, o);
        const int k2 = __shfl_xor_sync(FULL, bk, o);
        if (w2 < bw || (w2 == bw && k2 < bk)) {
          bw = w2;
          bk = k2;
        }
      }
    } else {
      const int src = nb ? __ffs((int)nb) - 1 : base;
      bw = __shfl_sync(FULL, bw, src);
      bk = __shfl_sync(FULL, bk, src);
    }
    const int mu = bk;
    const double dmin = bitsd(bw);
    const double tn = __dadd_rn(t, dmin);
    if (run) {
      if (mu == INT_MAX) {
        status = RT_TRAJ_ABSORBED;
        run = false;
      } else if (dbits(tn) > tend_bits) {
        status = RT_TRAJ_TEND;
        run = false;
      } else if (ev == A.max_events) {
        status = RT_TRAJ_MAX_EVENTS;
        run = false;
      }
    }
    // ---- the int32 range of the fired reaction's net change (a count past INT_MAX wraps below 0)
    int vb = 0, ve = 0;
    if (run) {
      vb = net.vp[mu];
      ve = net.vp[mu + 1];
    }
    bool over = false;
    for (int i = vb + sl; i < ve; i += G) {
      const int2 e = net.vl[i];
      over |= (int)((uint32_t)X[e.x] + (uint32_t)e.y) < 0;
    }
    if ((__ballot_sync(FULL, over) & segmask) != 0) {
      status = RT_TRAJ_OVERFLOW;
      run = false;
      ve = vb;
    }
    // ---- fire (segments still running)
    db = de = 0;
    double E = 0.0;
    if (run) {
      db = net.dptr[mu];
      de = net.dptr[mu + 1];
      while (gi < A.G && dbits(next_g) < dbits(tn)) {
        record(gi, true);
        ++gi;
        next_g = __dmul_rn(__ll2double_rn(gi), A.sample_dt);
      }
      tprev = t;
      t = tn;
      if (sl == 0) trace_event(A.out, j, ev, mu, tn);
      if (LL && sl == (ev & (G - 1)))
        ring = TD ? __dmul_rn(S.a[mu], __dadd_rn(1.0, __dmul_rn(net.beta[mu], t))) : S.a[mu];
      E = S.E[mu];
    }
    // the fired channel's increment: if it is used up, every lane draws one of its used-up ones, the fired
    // channel's owner that one
    if (__any_sync(FULL, dbits(E) < 0)) {
      if (stale) {
        const bool own = run && sl == (mu & (G - 1)) && ((stale >> (mu / G)) & 1u);
        const int r = own ? mu / G : __ffs((int)stale) - 1, k = sl + G * r;
        S.E[k] = exp1_draw(A.seed, g, (uint32_t)k, (uint32_t)(S.n[k] + 1), A.stream_id);
        stale &= ~(1u << r);
      }
      __syncwarp();
      if (run) E = S.E[mu];
    }
    __syncwarp();
    if (run) {
      for (int i = vb + sl; i < ve; i += G) {
        const int2 e = net.vl[i];
        X[e.x] += e.y;
      }
      if (sl == (mu & (G - 1))) {
        const double P = __dadd_rn(S.P[mu], E);  // Eq. 27
        S.P[mu] = P;
        S.b[mu].x = upper_P(P);
        S.E[mu] = -1.0;
        S.n[mu] += 1;
        stale |= 1u << (mu / G);
      }
      ++ev;
      dprev = dmin;
    }
    __syncwarp();
    if (LL) {
      const int cnt = (run && (ev & (G - 1)) == 0) ? G : 0;
      if (__any_sync(FULL, cnt != 0)) flush_ring(cnt);
    }
  }
  if (LL) flush_ring(live ? (ev & (G - 1)) : 0);

  const bool known = status == RT_TRAJ_TEND || status == RT_TRAJ_ABSORBED;
  if (A.out.loglik_dev || A.out.t_internal_dev) {
    if (live && known && tend_finite && !bad) {
      const double rest = __dsub_rn(A.t_end, t);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int k = sl + G * r;
        if (k < M) T[r] = __dadd_rn(T[r], __dmul_rn(S.a[k], TD ? tdep_integral(net.beta[k], t, rest) : rest));
      }
    }
    if (A.out.loglik_dev) {
      const double sT = warp_sum_T_in_order<R, G>(T, M, live);  // every lane takes part
      if (live && sl == 0) A.out.loglik_dev[j] = bad ? __longlong_as_double(0x7FF8000000000000ll) : __dsub_rn(ll, sT);
    }
    if (live && A.out.t_internal_dev)
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (sl + G * r < M) A.out.t_internal_dev[j * M + sl + G * r] = T[r];
  }
  if (!live) return;
  for (; gi < A.G; ++gi) record(gi, known);
  trace_tail(A.out, j, ev, sl, G);
  if (A.out.counts_dev)
    for (int k = sl; k < M; k += G) A.out.counts_dev[j * M + k] = S.n[k];
  if (A.out.x_final_dev)
    for (int s = sl; s < N; s += G) A.out.x_final_dev[j * N + s] = X[s];
  if (sl == 0) {
    if (A.out.n_events_dev) A.out.n_events_dev[j] = ev;
    if (A.out.status_dev) A.out.status_dev[j] = status;
    if (A.out.t_last_dev) A.out.t_last_dev[j] = t;
  }
}

}  // namespace rt

// rt_traj_block.cuh -- one thread block per trajectory.
//
// The NRRTA loop of Table 2 (Liu & Wang, arXiv:2103.00405) for networks of up to
// R * blockDim.x reactions: channel k belongs to thread k % B, slot k / B (Eq. 17-27).
// T_k is in registers; a_k and a pair of floats (upper bounds of P_k and 1 / a_k) in
// shared memory (or, where a block cannot hold them, in the thread's local memory), P_k
// and the increment drawn ahead for the channel's next firing, which an event reads for one
// or two channels, in local memory; firing counts, X, and a bitmap of the channels whose
// propensity must be recomputed in shared memory.  Per event three phases, a barrier after each:
//   Y: the last firing's owner adds its increment to P (Eq. 27); every T_k advances with the
//      pre-event a_k (Eq. 17) and gives a float interval of its waiting time; each lane
//      recomputes its marked propensities and their intervals (Eq. 1-2, one pass for all first
//      ones); the block minimum of the upper ends;
//   E: the channels whose interval reaches below that minimum are computed exactly (one or two
//      in the block) and listed with where their net change and dependents are stored;
//   X: every thread takes the smallest of the list, smallest index on ties (Eq. 25-26); the net
//      change is applied by one thread per species with the int32 range check (undone if it
//      fails), and the dependents are marked.
// The fired channel's next increment is drawn by its owner in two halves where the other warps
// wait anyway: the Philox block in phase E, its logarithm in phase X of the event after.
// What bounds it: the advance of T issues two FP64 warp instructions (16 cycles each) per 32
// channels and event, 2000 cycles per event at 2000 reactions; the rest of an event is latency
// (about as much), which the SM's other blocks fill.  Against P, T and a in (spilled) registers with
// every bound taken from them per event and one thread's draw on the path: 500 trajectories of 2000
// reactions, 5000 events each, 56 -> 31.8 ms; of 4096 reactions 114 -> 70 ms; 20 trajectories of 500
// reactions 37 -> 9.4 ms (with the block size by the number of trajectories); 512 networks of 4 to
// 4096 reactions in one batch 309 -> 210 ms.
#pragma once
#include <climits>

#include "rt_sim.cuh"

namespace rt {

struct BlockNet {
  int M, N;
  const int2 *rd;
  const double *c;
  const int *vp;
  const int2 *vl;
  const int *dptr;  // per reaction the channels its firing touches: dlist[dptr[k]..dptr[k+1])
  const int *dlist;
};

// a channel that may be the next to fire, and where its net change and dependents lie
struct __align__(16) BlockCand {
  long long w;
  int k, vb, ve, db, de;
  int owner;  // its thread and, from bit 16, its slot
};

// shared-memory scratch of one block trajectory
struct BlockScratch {
  double *a;       // [slots][B] propensities (SM)
  float2 *b;       // [slots][B] {P bound, 1 / a bound} (SM)
  BlockCand *cand; // [B]
  double *buf;     // [B]
  double *s_amu;   // propensity of the fired channel
  uint32_t *red;   // [warps] bits of each warp's smallest upper end
  int *s_over;     // set if the fired reaction would leave the int32 range
  int *s_cnt;      // entries of cand
  uint32_t *bm;    // [ceil(M/32)] channels whose propensity must be recomputed
  int *NK;         // [M] firing counts n_k
  int *X;          // [N]
};

// Candidates are usually one or two.  There are many where rates lie outside the float bounds' range (below 1e-37,
// above 1e35) or internal times are so far from 0 that the bounds are wide.  Above this number a warp reads the
// list together: 500 events of 64 trajectories of 3000 reactions, a third of them with rates of 1e-45, 3.7 ms where
// every thread reading all of it takes 13.5; with usual rates 500 trajectories of 2000 reactions 31.8 ms either way.
constexpr int kFewCand = 8;

__host__ __device__ inline size_t block_state_bytes(int M, int B) { return (size_t)((M + B - 1) / B) * B * 16; }

__host__ __device__ inline size_t block_scratch_bytes(int M, int N, int B) {
  return (size_t)B * (sizeof(BlockCand) + 8) + 16 + (size_t)(B / 32) * 4 + 8 + (size_t)((M + 31) / 32) * 4 +
         (size_t)M * 4 + (size_t)N * 4 + 64;
}

// state_bytes: what the SM arrays take at the start (0 without them)
__device__ inline BlockScratch carve_block_scratch(unsigned char *base, size_t state_bytes, int M, int N, int B) {
  BlockScratch s;
  s.a = (double *)base;
  s.b = (float2 *)(base + state_bytes / 2);
  s.cand = (BlockCand *)(base + state_bytes);
  s.buf = (double *)(s.cand + B);
  s.s_amu = s.buf + B;
  s.red = (uint32_t *)(s.s_amu + 1);
  s.s_over = (int *)(s.red + B / 32);
  s.s_cnt = s.s_over + 1;
  s.bm = (uint32_t *)(s.s_cnt + 1);
  s.NK = (int *)(s.bm + (M + 31) / 32);
  s.X = s.NK + M;
  return s;
}

// R: slots, ceil(M / B) with SM (the loops over slots then have no branch, so that the slots' 64-cycle FP64
// operations overlap; entries past M hold a = 0 and an interval at +inf), at least that without.
// SM: a and the float pairs in shared memory (else in the thread's local memory).
template <int R, bool LL, bool SM>
__device__ __forceinline__ void block_trajectory(const RunArgs &A, const BlockNet &net, const BlockScratch &S, const int64_t j,
                                 const int tend_finite) {
  const int tid = threadIdx.x, B = blockDim.x, lane = tid & 31, warp = tid >> 5, W = B >> 5;
  const int M = net.M, N = net.N;
  const int nbm = (M + 31) / 32;
  const uint64_t g = (uint64_t)(A.traj_offset + j);
  const int32_t *x0 = A.x0 + (A.per_traj_x0 ? j * (int64_t)N : 0);
  int *X = S.X;
  for (int s = tid; s < N; s += B) X[s] = x0[s];
  for (int w = tid; w < nbm; w += B) S.bm[w] = 0u;
  for (int k = tid; k < M; k += B) S.NK[k] = 0;
  if (tid == 0) *S.s_over = 0;
  __syncthreads();
  int badl = 0;
  for (int s = tid; s < N; s += B) badl |= X[s] < 0;
  const bool bad = __syncthreads_or(badl) != 0;
  auto xat = [&](int s) { return X[s]; };

  auto record = [&](int64_t gidx, bool known) {
    if (A.out.grid_dev) {
      int32_t *gp = A.out.grid_dev + (j * A.G + gidx) * N;
      for (int s = tid; s < N; s += B) gp[s] = known ? X[s] : -1;
    }
    if (!known || !A.out.grid_sum_dev) return;
    for (int s = tid; s < N; s += B) {
      const long long x = X[s];
      atomicAdd((unsigned long long *)(A.out.grid_sum_dev + gidx * N + s), (unsigned long long)x);
      if (A.out.grid_sumsq_dev)
        atomicAdd((unsigned long long *)(A.out.grid_sumsq_dev + gidx * N + s), (unsigned long long)(x * x));
    }
    if (tid == 0 && A.out.grid_count_dev) atomicAdd((unsigned long long *)(A.out.grid_count_dev + gidx), 1ull);
  };

  double T[R], P[R], En[R];
  float lo[R];
  double a_loc[SM ? 1 : R];
  float2 b_loc[SM ? 1 : R];
  auto a_ref = [&](int r) -> double & { return SM ? S.a[r * B + tid] : a_loc[SM ? 0 : r]; };
  auto b_ref = [&](int r) -> float2 & { return SM ? S.b[r * B + tid] : b_loc[SM ? 0 : r]; };
#pragma unroll
  for (int r = 0; r < R; ++r) T[r] = 0.0;
#pragma unroll 1
  for (int r = 0; r < R; ++r) {
    const int k = tid + B * r;
    P[r] = 1.0;
    {
      double av = 0.0;
      if (!bad && k < M) {
        P[r] = exp1_draw(A.seed, g, (uint32_t)k, 0u, A.stream_id);
        En[r] = exp1_draw(A.seed, g, (uint32_t)k, 1u, A.stream_id);
        av = propensity(net.rd[k], net.c[k], xat);
      }
      a_ref(r) = av;
      b_ref(r) = make_float2(upper_P(P[r]), inv_upper(av));
    }
  }
  int status = bad ? RT_TRAJ_BAD_X0 : RT_TRAJ_TEND;
  double t = 0.0, ll = 0.0, dmin = 0.0;
  bool fired = false;  // an event precedes this pass
  int owner = 0;       // thread and slot of the last fired channel
  int32_t ev = 0;
  int64_t gi = 0;
  double next_g = 0.0;
  const int64_t tend_bits = dbits(A.t_end);

  if (!bad) {
    for (;;) {
      // ---- phase Y
      if (fired && tid == (owner & 0xFFFF)) {  // Eq. 27
        const int rm = owner >> 16, k = tid + B * rm;
        const int32_t n = S.NK[k] + 1;
        S.NK[k] = n;
        P[rm] = __dadd_rn(P[rm], En[rm]);
        b_ref(rm).x = upper_P(P[rm]);
      }
      if (LL && fired && tid == 0) ll = __dadd_rn(ll, rt_ln(*S.s_amu));
      if (tid == 0) {
        *S.s_over = 0;
        *S.s_cnt = 0;
      }
      uint32_t todo = 0;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (warp + W * r < nbm) todo |= ((S.bm[warp + W * r] >> lane) & 1u) << r;
      const bool adv = dbits(dmin) != 0;
      float ub = __int_as_float(0x7F800000);
#pragma unroll
      for (int r = 0; r < R; ++r)
        {
          const double Tn = __dadd_rn(T[r], __dmul_rn(a_ref(r), dmin));
          T[r] = adv ? Tn : T[r];
          const float u = wait_interval(b_ref(r), T[r], lo[r]);
          ub = fminf(ub, (todo >> r) & 1u ? __int_as_float(0x7F800000) : u);
        }
      if (__any_sync(0xFFFFFFFFu, todo != 0)) {
        if (lane < R && warp + W * lane < nbm) S.bm[warp + W * lane] = 0u;  // this warp's words
        do {
          if (todo) {
            const int r = __ffs((int)todo) - 1, k = tid + B * r;
            const double av = propensity(net.rd[k], net.c[k], xat);
            a_ref(r) = av;
            const float2 q = make_float2(b_ref(r).x, inv_upper(av));
            b_ref(r).y = q.y;
            float l;
            ub = fminf(ub, wait_interval(q, pick<R>(T, r), l));
#pragma unroll
            for (int i = 0; i < R; ++i) lo[i] = i == r ? l : lo[i];
            todo &= todo - 1;
          }
        } while (__any_sync(0xFFFFFFFFu, todo != 0));
      }
      const uint32_t wub = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(fmaxf(ub, 0.0f)));
      if (lane == 0) S.red[warp] = wub;
      __syncthreads();
      // ---- phase E: the channels that reach below the block's smallest upper end, exactly; the last
      // firing's owner begins its next draw
      const float thr =
          interval_threshold(__uint_as_float(__reduce_min_sync(0xFFFFFFFFu, lane < W ? S.red[lane] : 0x7F800000u)));
      uint32_t need = 0;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (!(lo[r] > thr)) need |= 1u << r;
      if (need) {
        BlockCand e;
        e.w = kInfBits;
        e.k = INT_MAX;
        e.vb = e.ve = e.db = e.de = e.owner = 0;
        do {
          const int r = __ffs((int)need) - 1, k = tid + B * r;
          need &= need - 1;
          const double av = a_ref(r);
          if (dbits(av) == 0) continue;  // the padding past M too
          const int vb = net.vp[k], ve = net.vp[k + 1], db = net.dptr[k], de = net.dptr[k + 1];
          const long long wb = dbits(waiting_time(P[r], pick<R>(T, r), av));
          if (wb < e.w) {  // a thread's channels come in index order
            e.w = wb;
            e.k = k;
            e.vb = vb;
            e.ve = ve;
            e.db = db;
            e.de = de;
            e.owner = tid | (r << 16);
          }
        } while (need);
        if (e.k != INT_MAX) S.cand[atomicAdd(S.s_cnt, 1)] = e;
      }
      const bool drawing = fired && tid == (owner & 0xFFFF);
      const int rd = owner >> 16;
      uint64_t draw = 0;
      if (drawing) {
        const int k = tid + B * rd;
        draw = draw_bits(A.seed, g, (uint32_t)k, (uint32_t)S.NK[k] + 1u, A.stream_id);
      }
      __syncthreads();
      // ---- phase X: the smallest of the list (every thread the same decision)
      const int cnt = *S.s_cnt;
      if (cnt == 0) {
        status = RT_TRAJ_ABSORBED;
        break;
      }
      int ci = 0;
      long long bw = S.cand[0].w;
      int bk = S.cand[0].k;
      auto take = [&](int i) {
        const long long w2 = S.cand[i].w;
        const int k2 = S.cand[i].k;
        if (w2 < bw || (w2 == bw && k2 < bk)) {
          bw = w2;
          bk = k2;
          ci = i;
        }
      };
      if (cnt <= kFewCand) {
        for (int i = 1; i < cnt; ++i) take(i);
      } else {  // each lane its share
        for (int i = lane; i < cnt; i += 32) take(i);
        const int src = warp_argmin(bw, bk);
        bw = __shfl_sync(0xFFFFFFFFu, bw, src);
        bk = __shfl_sync(0xFFFFFFFFu, bk, src);
        ci = __shfl_sync(0xFFFFFFFFu, ci, src);
      }
      const double dnext = bitsd(bw);
      const double tn = __dadd_rn(t, dnext);
      if (dbits(tn) > tend_bits) {
        status = RT_TRAJ_TEND;
        break;
      }
      if (ev == A.max_events) {
        status = RT_TRAJ_MAX_EVENTS;
        break;
      }
      const int vb = S.cand[ci].vb, ve = S.cand[ci].ve;
      if (gi < A.G && dbits(next_g) < dbits(tn)) {
        // grid samples from the pre-event X, after the range check (an overflowing event
        // records nothing); X is only read until the barrier below
        bool over = false;
        for (int i = vb; i < ve; ++i) {
          const int2 e = net.vl[i];
          over |= (int)((uint32_t)X[e.x] + (uint32_t)e.y) < 0;
        }
        if (over) {
          status = RT_TRAJ_OVERFLOW;
          break;
        }
        while (gi < A.G && dbits(next_g) < dbits(tn)) {
          record(gi, true);
          ++gi;
          next_g = __dmul_rn(__ll2double_rn(gi), A.sample_dt);
        }
        __syncthreads();
      }
      for (int i = vb + tid; i < ve; i += B) {
        const int2 e = net.vl[i];
        const int nx = (int)((uint32_t)X[e.x] + (uint32_t)e.y);
        if (nx < 0) *S.s_over = 1;  // a count past INT_MAX wraps below 0
        X[e.x] = nx;
      }
      for (int q = S.cand[ci].db + tid; q < S.cand[ci].de; q += B) {
        const int ch = net.dlist[q];
        atomicOr(&S.bm[ch >> 5], 1u << (ch & 31));
      }
      if (drawing) En[rd] = exp1_from_bits(draw);
      owner = S.cand[ci].owner;
      if (LL && tid == (owner & 0xFFFF)) *S.s_amu = a_ref(owner >> 16);
      __syncthreads();
      if (*S.s_over) {  // undo: the event does not fire
        for (int i = vb + tid; i < ve; i += B) {
          const int2 e = net.vl[i];
          X[e.x] = (int)(uint32_t)((uint32_t)X[e.x] - (uint32_t)e.y);
        }
        status = RT_TRAJ_OVERFLOW;
        break;
      }
      t = tn;
      if (tid == 0) trace_event(A.out, j, ev, bk, tn);
      ++ev;
      dmin = dnext;
      fired = true;
    }
  }

  __syncthreads();
  const bool known = status == RT_TRAJ_TEND || status == RT_TRAJ_ABSORBED;
  for (; gi < A.G; ++gi) record(gi, known);
  if (A.out.loglik_dev || A.out.t_internal_dev) {
    if (known && tend_finite && !bad) {
      const double rest = __dsub_rn(A.t_end, t);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (tid + B * r < M) T[r] = __dadd_rn(T[r], __dmul_rn(a_ref(r), rest));
    }
    if (A.out.t_internal_dev)
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (tid + B * r < M) A.out.t_internal_dev[j * M + tid + B * r] = T[r];
    if (A.out.loglik_dev) {
      double sT = 0.0;  // sum_k T_k in k order, B values at a time through shared memory
#pragma unroll
      for (int r = 0; r < R; ++r) {
        S.buf[tid] = T[r];
        __syncthreads();
        if (tid == 0)
          for (int l = 0; l < B && l + B * r < M; ++l) sT = __dadd_rn(sT, S.buf[l]);
        __syncthreads();
      }
      if (tid == 0) A.out.loglik_dev[j] = bad ? __longlong_as_double(0x7FF8000000000000ll) : __dsub_rn(ll, sT);
    }
  }
  if (A.out.counts_dev)
    for (int k = tid; k < M; k += B) A.out.counts_dev[j * M + k] = S.NK[k];
  if (A.out.x_final_dev)
    for (int s = tid; s < N; s += B) A.out.x_final_dev[j * N + s] = X[s];
  trace_tail(A.out, j, ev, tid, B);
  if (tid == 0) {
    if (A.out.n_events_dev) A.out.n_events_dev[j] = ev;
    if (A.out.status_dev) A.out.status_dev[j] = status;
    if (A.out.t_last_dev) A.out.t_last_dev[j] = t;
  }
  __syncthreads();
}

}  // namespace rt

// rt_lane.cu -- few trajectories of a small network (M <= 16 reactions, N <= 32 species): a warp
// per trajectory, a lane per channel.
//
// One thread per trajectory (rt_small.cu, rt_thread.cu) is the better use of the chip once there
// are enough trajectories to fill it.  With few, a run takes as long as its events one after the
// other, and a thread's event is a chain of some 700 instructions: each channel in turn, then the
// draw, then each propensity.  Here a warp works on one event:
//   - lane l < M holds channel l's P, T, a and the counts of its two reactants; lane s < N holds
//     X_s.  The change of all three by a firing is one 16-byte shared-memory load (table [mu][lane]).
//   - the next D = 32 / MP Exp(1) increments of every channel (MP: M rounded up to a power of two)
//     are drawn ahead, one per lane: increment n of channel k in lane k + MP ((n - 1) % D).  When a
//     used-up one is needed, every used-up lane draws its next in the same pass, so a pass serves
//     about as many events as there are lanes.  (E_n depends on the seed, the trajectory, the channel
//     and n only.)
//   - the winner comes from float estimates of the waiting times by a warp minimum (redux) and a vote;
//     its exact waiting time, which only t and the T_k need, is computed while the winner's net change
//     and the new propensities are.  An event whose two smallest estimates are within 2^-17, or whose
//     values are outside the estimates' range, takes the exact minimum over all lanes.
// What bounds it is the latency of one event, some 210 instructions, of which the chain
// P - T, quotient, T + a dt (64 cycles per FP64 operation, 200 for the quotient) is about 450 cycles:
// 0.5 us per event (one thread per trajectory: 1.8 us; 2.8 us before its arithmetic was changed).
// The operations and their order per channel are those of the other mappings: the same bits.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>

#include "rt_sim.cuh"

namespace rt {

constexpr int kLaneMaxM = 16, kLaneMaxN = 32;

// IMUL: the propensity's product on the integer pipe.
template <int MP, bool LL, bool IMUL>
__global__ void __launch_bounds__(128) k_ens_lane(const RunArgs A, const int tend_finite) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned FULL = 0xFFFFFFFFu;
  constexpr uint32_t D = 32 / MP;  // increments of a channel held ahead
  int4 *tab = (int4 *)smem;        // [M][32]: change of {X_lane, first and second factor of lane's propensity}
  const DevNet &net = A.net;
  const int M = net.M, N = net.N;
  const int lane = threadIdx.x & 31;
  const int2 rd = lane < M ? net.rdesc[lane] : make_int2(RD_NONE, RD_UNI);
  const bool dimer = rd.x >= 0 && rd.y == RD_DIMER;
  const int sp1 = dimer ? rd.x : rd.y;  // species of the second factor (dimer: x (x - 1) / 2)
  for (int mu = threadIdx.x >> 5; mu < M; mu += blockDim.x >> 5) {
    int4 e = make_int4(0, 0, 0, 0);
    for (int i = net.vptr[mu]; i < net.vptr[mu + 1]; ++i) {
      const int2 v = net.vlist[i];
      if (v.x == lane) e.x = v.y;
      if (rd.x >= 0 && v.x == rd.x) e.y = v.y;
      if (rd.x >= 0 && sp1 >= 0 && v.x == sp1) e.z = v.y;
    }
    tab[mu * 32 + lane] = e;
  }
  __syncthreads();
  const int64_t j = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= A.n_traj) return;  // whole warps; no block barrier below

  const uint64_t g = (uint64_t)(A.traj_offset + j);
  const int32_t *x0 = A.x0 + (A.per_traj_x0 ? j * (int64_t)N : 0);
  int X = lane < N ? x0[lane] : 0;
  const bool bad = __any_sync(FULL, X < 0);
  // the two factors of h_k: x[s0], x[s1] (bimolecular), x[s0], 1 (unimolecular), 1, 1 (no reactant),
  // x[s0], x[s0] - 1 and a halving (dimer)
  int xa = rd.x >= 0 ? x0[rd.x] : 1;
  int xb = rd.x >= 0 && sp1 >= 0 ? x0[sp1] - (dimer ? 1 : 0) : 1;
  const double c = lane < M ? net.c[lane] : IMUL ? 1.0 : 0.0;
  const int half = dimer ? 1 : 0;
  auto prop = [&](int f0, int f1) {
    const int64_t h = ((int64_t)f0 * f1) >> half;
    if (!IMUL) return __dmul_rn(c, __ll2double_rn(h));
    const double v = mul_rn_pos_u32(c, h);
    return lane < M ? v : 0.0;
  };

  double P = 0.0, T = 0.0, a = 0.0, E = 0.0;
  int32_t n = 0;                                  // firings of this lane's channel
  uint32_t nd = 1 + (uint32_t)lane / MP;          // index of the increment in E
  const uint32_t dk = (uint32_t)lane & (MP - 1);  // and its channel
  int status = RT_TRAJ_TEND;
  double t = 0.0, ll = 0.0;
  int32_t ev = 0;
  int64_t gi = 0;
  double next_g = 0.0;
  double ring = 0.0;  // with the likelihood: a_mu of event (ev & ~31) + lane

  auto record = [&](int64_t gidx, bool known) {
    if (A.out.grid_dev && lane < N) A.out.grid_dev[(j * A.G + gidx) * N + lane] = known ? X : -1;
    if (!known || !A.out.grid_sum_dev) return;
    if (lane < N) {
      const long long x = X;
      atomicAdd((unsigned long long *)(A.out.grid_sum_dev + gidx * N + lane), (unsigned long long)x);
      if (A.out.grid_sumsq_dev)
        atomicAdd((unsigned long long *)(A.out.grid_sumsq_dev + gidx * N + lane), (unsigned long long)(x * x));
    }
    if (lane == 0 && A.out.grid_count_dev) atomicAdd((unsigned long long *)(A.out.grid_count_dev + gidx), 1ull);
  };
  auto flush_ring = [&](int cnt) {  // ll += ln a_mu of the cnt buffered events, in event order
    double v = 0.0;
    if (lane < cnt) v = rt_ln(ring);
    for (int i = 0; i < cnt; ++i) ll = __dadd_rn(ll, __shfl_sync(FULL, v, i));
  };

  if (bad) {
    status = RT_TRAJ_BAD_X0;
  } else {
    if (lane < M) P = exp1_draw(A.seed, g, (uint32_t)lane, 0u, A.stream_id);
    a = prop(xa, xb);
    if (dk < (uint32_t)M) E = exp1_draw(A.seed, g, dk, nd, A.stream_id);
    unsigned used = 0;  // lanes whose increment is used up (the same in every lane)
    const int64_t tend_bits = dbits(A.t_end);
    const int32_t max_ev = A.max_events;
    const int32_t ntrace = (int32_t)min(A.out.trace_len, (int64_t)INT_MAX);
    // the test at the end of an event is taken when t passes tlim: t_end or the next grid time
    int64_t tlim = min(tend_bits, A.G > 0 ? dbits(next_g) : kInfBits);
    float y = mant_rcp(a);
    int forced = -1;  // the winner, when the exact comparison had to name it
    for (;;) {
      // One event in one straight run of instructions up to the single test below, so that the
      // independent chains (the quotient, the net change and the new propensities, the 64-cycle FP64
      // operations) overlap; nothing of the state changes before that test.
      // Eq. 25-26: the smallest waiting time (smallest index on ties)
      const double rem = __dsub_rn(P, T);
      const uint32_t hi = (uint32_t)__double2hiint(rem), ah = (uint32_t)__double2hiint(a);
      const bool act = dbits(a) != 0;
      // estimate: the float below rem, over a's exponent and (within 2^-22) its significand
      const float ia = __uint_as_float(__float_as_uint(y) - (ah >> 20 << 23) + (1023u << 23));
      const bool in = hi - (897u << 20) < (253u << 20) && ah - (900u << 20) < (240u << 20);
      uint32_t e = in ? __float_as_uint(__uint_as_float(hi * 8u - 0xC0000000u) * ia) : 0u;
      e = act ? e : 0x7F800000u;
      const float m1 = __uint_as_float(__reduce_min_sync(FULL, e));
      const unsigned close = __ballot_sync(FULL, __uint_as_float(e) <= m1 * 1.00000763f);
      const bool sure = m1 >= 1e-30f && m1 < 1e30f && (close & (close - 1)) == 0;
      const int mu = forced >= 0 ? forced : __ffs(close) - 1;
      const int4 d = tab[mu * 32 + lane];
      const double w = act ? (dbits(rem) > 0 ? div_rn_pos(rem, a, y) : 0.0) : bitsd(kInfBits);
      const double dt = __shfl_sync(FULL, w, mu);
      const uint32_t nmu = (uint32_t)__shfl_sync(FULL, n, mu);      // firings before this one
      const int src = mu + MP * (int)(nmu & (D - 1));               // its next increment (Eq. 27)
      const double Emu = __shfl_sync(FULL, E, src);
      const double tn = __dadd_rn(t, dt);
      const double Tn = __dadd_rn(T, __dmul_rn(a, dt));             // Eq. 17 (a = 0 past M)
      const double Pn = __dadd_rn(P, Emu);
      const int Xn = (int)((uint32_t)X + (uint32_t)d.x);            // past INT_MAX it wraps below 0
      const int xan = (int)((uint32_t)xa + (uint32_t)d.y), xbn = (int)((uint32_t)xb + (uint32_t)d.z);
      const double an = prop(xan, xbn);
      const float yn = mant_rcp(an);
      const bool over = __any_sync(FULL, Xn < 0);
      if ((!sure && forced < 0) || dbits(tn) > tlim || ev == max_ev || over || ev < ntrace) {
        if (!sure && forced < 0) {
          const uint32_t wh = (uint32_t)__double2hiint(w);
          const uint32_t mh = __reduce_min_sync(FULL, wh);
          const uint32_t wl = wh == mh ? (uint32_t)__double2loint(w) : 0xFFFFFFFFu;
          const uint32_t ml = __reduce_min_sync(FULL, wl);
          forced = __ffs(__ballot_sync(FULL, wh == mh && wl == ml)) - 1;
          if (mh < 0x7FF00000u) continue;  // a finite waiting time
          status = RT_TRAJ_ABSORBED;
          break;
        }
        if (dbits(tn) > tend_bits) {
          status = RT_TRAJ_TEND;
          break;
        }
        if (ev == max_ev) {
          status = RT_TRAJ_MAX_EVENTS;
          break;
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
        tlim = min(tend_bits, gi < A.G ? dbits(next_g) : kInfBits);
        if (lane == 0) trace_event(A.out, j, ev, mu, tn);
      }
      forced = -1;
      if (LL) {
        const double amu = __shfl_sync(FULL, a, mu);
        if (lane == (ev & 31)) ring = amu;
      }
      ++ev;
      t = tn;
      T = Tn;
      if (lane == mu) {
        P = Pn;
        n += 1;
      }
      X = Xn;
      xa = xan;
      xb = xbn;
      a = an;
      y = yn;
      // every channel's next increment is kept fresh
      used |= 1u << src;
      if ((used >> (mu + MP * (int)((nmu + 1) & (D - 1)))) & 1u) {
        if ((used >> lane) & 1u) {
          nd += D;
          E = exp1_draw(A.seed, g, dk, nd, A.stream_id);
        }
        used = 0;
      }
      if (LL && (ev & 31) == 0) flush_ring(32);
    }
  }
  if (LL) flush_ring(ev & 31);

  const bool known = status == RT_TRAJ_TEND || status == RT_TRAJ_ABSORBED;
  for (; gi < A.G; ++gi) record(gi, known);
  if (A.out.loglik_dev || A.out.t_internal_dev) {
    if (known && tend_finite) T = __dadd_rn(T, __dmul_rn(a, __dsub_rn(A.t_end, t)));
    if (A.out.t_internal_dev && lane < M) A.out.t_internal_dev[j * M + lane] = T;
    if (A.out.loglik_dev) {
      double sT = 0.0;
      for (int k = 0; k < M; ++k) sT = __dadd_rn(sT, __shfl_sync(FULL, T, k));
      if (lane == 0) A.out.loglik_dev[j] = bad ? __longlong_as_double(0x7FF8000000000000ll) : __dsub_rn(ll, sT);
    }
  }
  if (A.out.counts_dev && lane < M) A.out.counts_dev[j * M + lane] = n;
  if (A.out.x_final_dev && lane < N) A.out.x_final_dev[j * N + lane] = X;
  trace_tail(A.out, j, ev, lane, 32);
  if (lane == 0) {
    if (A.out.n_events_dev) A.out.n_events_dev[j] = ev;
    if (A.out.status_dev) A.out.status_dev[j] = status;
    if (A.out.t_last_dev) A.out.t_last_dev[j] = t;
  }
}

// Up to 8 warps per SM the FP64 pipe is idle most of the time and its product (two instructions of 64
// cycles beside the quotient) is the shorter way to a propensity; above, the pipe fills up (an event
// issues eight FP64 instructions, 16 cycles each) and the integer product is used (Lotka-Volterra to
// t = 0.3, FP64 / integer: 64 trajectories 5.1 / 5.5 ms, 1000 6.1 / 6.3 ms, 2000 9.9 / 8.2 ms).
constexpr int64_t kLaneFp64Traj = 152 * 8;

// Where the lane kernel is used (when the caller leaves the mapping to the library): below the
// ensemble sizes at which one thread per trajectory overtakes it.  Measured, lane / thread: Lotka-Volterra
// 64 trajectories 5.1 / 17.0 ms, 3000 9.8 / 17.9 ms, 8000 25.8 / 18.3 ms; birth-death 64 0.62 / 1.53 ms,
// 3000 1.18 / 1.60 ms, 4000 1.65 / 1.64 ms; 12 reactions 64 1.0 / 8.0 ms, 8000 4.7 / 8.1 ms,
// 16000 8.6 / 8.6 ms; 16 reactions 8000 16.7 / 27 ms, 16000 30 / 28 ms.  A thread's event takes longer with M, a
// warp's does not.  Time of the thread kernel over the lane kernel's, three networks each, at 152 x 64 / 152 x 72
// trajectories: 5 reactions 0.90, 1.10, 1.07 / 0.80, 0.98, 0.91; 6 reactions 1.15, 1.27, 1.06 / 1.02, 1.11, 0.92;
// 7 reactions 1.08, 1.19, 1.17 / 0.95, 1.06, 1.03; 8 and 9 at least 1.21 / 1.08.
bool lane_mapping_fits(const DevNet &net, int64_t n_traj) {
  return net.M <= kLaneMaxM && net.N <= kLaneMaxN && n_traj <= 152 * (net.M <= 4 ? 24 : net.M == 5 ? 64 : 72);
}

template <int MP>
static cudaError_t launch_lane_m(const RunArgs &a, cudaStream_t s) {
  // a warp per SM as long as there are SMs left, then four warps per block
  const int B = a.n_traj <= 152 * 4 ? 32 : 128;
  const unsigned grid = (unsigned)((a.n_traj + B / 32 - 1) / (B / 32));
  const int tf = std::isfinite(a.t_end) ? 1 : 0;
  const size_t smem = (size_t)a.net.M * 32 * sizeof(int4);  // at most 8 KB
  const bool imul = a.n_traj > kLaneFp64Traj;
  auto kern = a.out.loglik_dev ? (imul ? k_ens_lane<MP, true, true> : k_ens_lane<MP, true, false>)
                               : (imul ? k_ens_lane<MP, false, true> : k_ens_lane<MP, false, false>);
  kern<<<grid, B, smem, s>>>(a, tf);
  return cudaGetLastError();
}

int launch_lane_mapping(const RunArgs &a, cudaStream_t s) {
  if (a.n_traj == 0) return RT_OK;
  const int M = a.net.M;
  const cudaError_t e = M <= 4 ? launch_lane_m<4>(a, s) : M <= 8 ? launch_lane_m<8>(a, s) : launch_lane_m<16>(a, s);
  if (e != cudaSuccess) return set_error(RT_ERR_CUDA, "lane kernel launch: %s", cudaGetErrorString(e));
  return RT_OK;
}

}  // namespace rt

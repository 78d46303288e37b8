// rt_lazy.cu -- large networks in the absolute-time form: a thread-block cluster per
// trajectory, the argmin kept in a min-tree, only the touched channels updated per event.
//
// The method in its absolute-time ("lazy") form, the Gibson-Bruck next reaction method
// with the dependency graph the paper describes (Sec. 5; Eq. 17, 24-27 in internal
// times): every channel keeps P_k, T_k (its internal time up to the real time s_k of
// its last update), a_k and its absolute firing time tau_k = s_k + (P_k - T_k) / a_k.
// An event at t = tau_mu touches only mu and the channels that read a species the
// event changed: T_k += a_k (t - s_k), s_k = t, P_mu += E (Eq. 27), a_k = c_k h_k(X)
// (Eq. 1-2), tau_k recomputed.  Every other tau_k stays as it is, so an event costs a
// few hundred channel updates instead of a pass over all M channels.
//
// The argmin over tau is the paper's "binary tree searching" of the next reaction
// (Sec. 6) in GPU form: the trajectory's channels are split into C contiguous slices,
// one per CTA of a thread-block cluster; a CTA keeps, in shared memory, the minimum
// (tau, k) of every group of 32 consecutive channels of its slice.  Per event a CTA
//   1. reduces its group minima to its slice minimum (a thread reads its groups again only
//      when one of them changed, a warp its candidate's dependency record when that changed),
//   2. posts it with the record into every CTA's mailbox (distributed shared memory, words that
//      carry their own tags, no ordering between them) and polls its own mailbox (bounded: after
//      spin_limit polls the trajectory ends with RT_TRAJ_TIMEOUT) -- every thread of every CTA
//      then takes the same decision from the same C entries,
//   3. updates the touched channels of its slice (from the species -> readers lists, packed
//      to full warps; the counts after the event are the old ones plus the net change, so X is
//      written behind a later barrier), while idle warps prefetch what the slice would read for
//      the candidate that came second, the likeliest to fire next,
//   4. updates the minima of the 32-channel groups that hold a touched channel (one thread per
//      group; a group whose minimum was touched re-reads its untouched channels, one warp each).
// What bounds it is latency: an event is a chain of memory (1500 cycles a miss; the records of 16
// trajectories of 10^6 channels are 512 MB), barriers and 64-cycle FP64 operations.  It moves 153 KB per
// event (104 KB before the prefetch for the second candidate; 42 KB by count), 6.6 % of the memory's rate.
// Per event at that size 7.9 us when one thread polled, decided and wrote the decision
// for the others and every touched channel was loaded in three dependent steps and divided on the
// FP64 pipe; 6.8 us without those, 6.4 us with packed lists, 5.5 us with the prefetch.
// Ties go to the smallest index at every level, so the minimum is the exact one.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>

#include "rt_sim.cuh"

namespace cg = cooperative_groups;

namespace rt {

constexpr int kLazyThreads = 512;
constexpr int kLazyWarps = kLazyThreads / 32;
constexpr int kLazyMaxC = 16;
constexpr int kLazyMaxVlen = 16;  // net-change entries of one reaction kept in shared memory

// one channel's state; 32 bytes so a touched channel is one sector
struct __align__(32) ChanRec {
  double P;  // internal time of the next firing
  double T;  // internal time accounted up to s
  double s;  // real time of the last update
  double a;  // propensity since s
};

constexpr int kPostWarp = kLazyWarps - 1;         // the slice minimum, the posts, prefetches, and the draws
constexpr int kFireTid = (kLazyWarps - 2) * 32;    // lane 0 of warp 14 updates the fired channel

// A mailbox slot: the posting CTA's slice minimum for one event and its dependency record
// (DevNet::vdep), as 64-bit words that each carry a tag saying which use of the slot they belong to,
// so a post needs no ordering between its stores (a releasing store waits for the acknowledgement of
// those before it, a round trip between SMs) and the reader takes each word as it comes.  The tag is a
// bit that is 0 in the data (the sign of a time or propensity >= 0, bit 31 of an offset or a length) and
// alternates from one use of a slot to the next; word 1 holds the event's number instead.
//   0: tau  1: event << 32 | channel  2: propensity  3-6: net change i, reader list begin i << 32
//   7, 8: reader list lengths 2i, 2i + 1 << 32
constexpr int kMailWords = 9;
struct __align__(16) Mail {
  unsigned long long word[kMailWords + 1];
};
__device__ __forceinline__ unsigned long long mail_tag(unsigned seq) {
  // a slot's words alternate with seq / 2 (two slots by the parity of seq); the first use has tag 1
  const unsigned long long t = ((seq - 1) >> 1) & 1 ? 0ull : 1ull;
  return t << 63;
}

struct LazyArgs {
  RunArgs r;
  int C;              // CTAs per trajectory (cluster size)
  int64_t Ms;         // row stride of CH / TAU / ENX / NK (multiple of 32 * C)
  int64_t chunk;      // channels per CTA slice (multiple of 32)
  ChanRec *CH;
  double *TAU;
  double *ENX;        // each channel's next Exp(1) increment, drawn ahead of its firing
  int32_t *NK;
  int cap;            // entries of one event's list of touched channels, at most
  int compact;        // 1: the list also holds a channel once per reader list it is found in
  int sptr_smem;      // 1: the species -> readers offsets are copied to shared memory
  int tend_finite;
  int want_T;         // t_internal or loglik requested
  long long spin_limit;
};

// Absolute firing time of a channel updated at real time su (Eq. 25 in absolute form).
__device__ __forceinline__ double lazy_tau(double P, double T, double a, double su) {
  if (dbits(a) == 0) return bitsd(kInfBits);
  const double rem = __dsub_rn(P, T);
  return __dadd_rn(su, waiting_time_rem(rem, a));
}

__global__ void k_lazy_init(const LazyArgs L) {
  const RunArgs &r = L.r;
  const int64_t total = r.n_traj * L.Ms;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = i / L.Ms;
    const int64_t k = i - j * L.Ms;
    ChanRec c;
    c.T = 0.0;
    c.s = 0.0;
    c.P = 0.0;
    c.a = 0.0;
    double tau = bitsd(kInfBits), enx = 0.0;
    if (k < r.net.M) {
      const int32_t *x0 = r.x0 + (r.per_traj_x0 ? j * r.net.N : 0);
      const uint64_t g = (uint64_t)(r.traj_offset + j);
      c.P = exp1_draw(r.seed, g, (uint32_t)k, 0u, r.stream_id);
      enx = exp1_draw(r.seed, g, (uint32_t)k, 1u, r.stream_id);
      c.a = propensity<false>(r.net.rdesc[k], r.net.c[k], [&](int s) { return x0[s]; });
      tau = lazy_tau(c.P, 0.0, c.a, 0.0);
    }
    L.CH[i] = c;
    L.TAU[i] = tau;
    L.ENX[i] = enx;
    L.NK[i] = 0;
  }
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(addr), "r"(rank));
  return out;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, unsigned long long v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

__device__ __forceinline__ unsigned long long ld_mail(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(smem_addr(p)) : "memory");
  return v;
}

__device__ __forceinline__ bool lex_less(long long w1, int k1, long long w2, int k2) {
  return w1 < w2 || (w1 == w2 && k1 < k2);
}

// a warp's candidate for the slice minimum; its dependency record is copied here asynchronously when
// the candidate changes, and is complete from the event after that (epoch < seq)
struct __align__(16) PostStage {
  int4 v, rb, rl;
  long long w;
  int k;
  unsigned epoch;
};

// the fired reaction's net change and reader lists where DevNet::vdep does not hold them
struct LazyLists {
  int2 vl[kLazyMaxVlen];
  int ofs[kLazyMaxVlen + 1];  // prefix offsets into the changed species' reader lists
  int beg[kLazyMaxVlen];
  int vlen;
};

__device__ __forceinline__ void copy16_async(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The next number of a shared counter, one atomic operation for the lanes that ask together.
__device__ __forceinline__ int take_number(int *ctr) {
  const unsigned m = __activemask();
  const int lane = threadIdx.x & 31, lead = __ffs((int)m) - 1;
  int b = 0;
  if (lane == lead) b = atomicAdd(ctr, __popc(m));
  return __shfl_sync(m, b, lead) + __popc(m & ((1u << lane) - 1u));
}

// VD: the network has dependency records (DevNet::vdep).
template <bool LL, bool VD>
__global__ void __launch_bounds__(kLazyThreads, 1) k_lazy(const LazyArgs L) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Mail mbox[2][kLazyMaxC];
  __shared__ PostStage red[kLazyWarps];  // each warp's candidate for the slice minimum
  __shared__ LazyLists lists;
  __shared__ uint32_t s_dirty[kLazyWarps];  // per warp the threads one of whose groups changed its minimum
  __shared__ int s_bad, s_ntouch, s_nrel, s_ngl, s_ok, s_pend_k, s_pend_n;

  cg::cluster_group cluster = cg::this_cluster();
  const RunArgs &r = L.r;
  const int M = r.net.M, N = r.net.N;
  const int C = L.C;
  const int c = (int)cluster.block_rank();
  const int64_t j = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t k0 = (int64_t)c * L.chunk;
  const int64_t k1 = min((int64_t)M, k0 + L.chunk);
  const int ng = (int)(L.chunk / 32);  // 32-channel groups of this slice (the last CTA's may run past M)
  const int cap = L.cap;

  // shared memory: per group its minimum (tau bits, channel) and the head of this event's list
  // of its touched channels; the touched channels of an event with their new firing times and
  // list links; the touched groups; per reloaded group its touched-channel minimum and mask; X;
  // species offsets
  long long *gw = (long long *)smem;
  long long *tw = gw + ng;
  long long *rcw = tw + cap;
  int *gk = (int *)(rcw + cap);
  int *ghead = gk + ng;
  int *tk = ghead + ng;
  int *tnext = tk + cap;
  int *glist = tnext + cap;
  int *rq = glist + cap;
  int *rck = rq + cap;
  uint32_t *rmask = (uint32_t *)(rck + cap);
  int *Xs = (int *)(rmask + cap);
  int *sp = Xs + N;
  const int *sptr = L.sptr_smem ? sp : r.net.sptr;

  ChanRec *CH = L.CH + j * L.Ms;
  double *TAU = L.TAU + j * L.Ms;
  double *ENX = L.ENX + j * L.Ms;
  int32_t *NK = L.NK + j * L.Ms;
  const uint64_t g = (uint64_t)(r.traj_offset + j);
  const int32_t *x0 = r.x0 + (r.per_traj_x0 ? j * N : 0);

  for (int i = tid; i < 2 * kLazyMaxC; i += blockDim.x) {
    Mail &m = mbox[i / kLazyMaxC][i % kLazyMaxC];
    for (int n = 0; n <= kMailWords; ++n) m.word[n] = 0ull;
  }
  if (tid == 0) {
    s_bad = 0;
    s_ntouch = 0;
    s_nrel = 0;
    s_ngl = 0;
    s_pend_k = -1;
    s_pend_n = 0;
  }
  if (tid < kLazyWarps) s_dirty[tid] = 0xFFFFFFFFu;
  __syncthreads();
  for (int s = tid; s < N; s += blockDim.x) {
    const int v = x0[s];
    Xs[s] = v;
    if (v < 0) s_bad = 1;
  }
  if (L.sptr_smem)
    for (int s = tid; s <= N; s += blockDim.x) sp[s] = r.net.sptr[s];
  for (int q = tid; q < ng; q += blockDim.x) ghead[q] = -1;
  // group minima of the slice from the initial firing times
  for (int q = warp; q < ng; q += kLazyWarps) {
    const int64_t k = k0 + (int64_t)q * 32 + lane;
    long long w = kInfBits;
    int kk = INT_MAX;
    if (k < k1) {
      w = dbits(TAU[k]);
      kk = (int)k;
    }
    if (lane == warp_argmin(w, kk)) {
      gw[q] = w;
      gk[q] = kk;
    }
  }
  __syncthreads();
  cluster.sync();  // every mailbox is zeroed before any CTA posts into it
  const bool bad = s_bad != 0;

  const uint32_t mb_local = smem_addr(&mbox[0][0]);
  double t = 0.0, ll = 0.0;
  int32_t ev = 0;
  int status = bad ? RT_TRAJ_BAD_X0 : RT_TRAJ_TEND;
  unsigned int seq = 0;  // posts so far
  int64_t gi = 0;
  double next_g = 0.0;
  const int64_t tend_bits = dbits(r.t_end);
  long long mw = kInfBits;  // the minimum of this thread's groups q = tid + 512 i
  int mk = INT_MAX;
  int cand_k = -1;  // this warp's candidate whose record red[warp] holds

  auto record = [&](int64_t gidx, bool known) {  // CTA 0, all threads
    if (r.out.grid_dev) {
      int32_t *gp = r.out.grid_dev + (j * r.G + gidx) * N;
      for (int s = tid; s < N; s += blockDim.x) gp[s] = known ? Xs[s] : -1;
    }
    if (r.out.grid_sum_dev && known) {
      for (int s = tid; s < N; s += blockDim.x) {
        const long long x = Xs[s];
        atomicAdd((unsigned long long *)(r.out.grid_sum_dev + gidx * N + s), (unsigned long long)x);
        if (r.out.grid_sumsq_dev)
          atomicAdd((unsigned long long *)(r.out.grid_sumsq_dev + gidx * N + s), (unsigned long long)(x * x));
      }
      if (tid == 0 && r.out.grid_count_dev) atomicAdd((unsigned long long *)(r.out.grid_count_dev + gidx), 1ull);
    }
  };
  // a touched channel of the slice and its new firing time join this event's list and the
  // list of its group; the first one of a group lists the group
  auto touch = [&](int64_t k, long long w, int i) {
    tk[i] = (int)k;
    tw[i] = w;
    const int q = (int)((k - k0) >> 5);
    const int nx = atomicExch(&ghead[q], i);
    tnext[i] = nx;
    if (nx < 0) glist[take_number(&s_ngl)] = q;
  };
  // group q's minimum changed: the thread that holds it in its own minimum takes it up
  auto set_group = [&](int q, long long w, int k) {
    gw[q] = w;
    gk[q] = k;
    atomicOr(&s_dirty[(q & (kLazyThreads - 1)) >> 5], 1u << (q & 31));
  };

  // a posted record: net-change words, list begins, prefix offsets of the list lengths (0 where unused)
  auto unpack = [&](const unsigned long long *m, int (&vw)[4], int (&lb)[4], int (&lo)[5]) {
    lo[0] = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned long long x = ld_mail(m + 3 + i), y = ld_mail(m + 7 + i / 2);
      vw[i] = (int)(uint32_t)x;
      lb[i] = (int)((x >> 32) & 0x7FFFFFFFu);
      lo[i + 1] = lo[i] + (vpack_delta(vw[i]) != 0 ? (int)((i & 1 ? y >> 32 : y) & 0x7FFFFFFFu) : 0);
    }
  };
  // where entry e of the concatenated reader lists lies
  auto entry = [&](int e, const int (&lb)[4], const int (&lo)[5], int &li) {
    int at = lb[0] + e;
    li = 0;
#pragma unroll
    for (int i = 1; i < 4; ++i)
      if (e >= lo[i]) {
        li = i;
        at = lb[i] + (e - lo[i]);
      }
    return at;
  };

  if (!bad) {
    for (;;) {
      // ---- 1. the slice minimum.  Each thread keeps the minimum of its groups and reads them again only
      // when one changed; each warp its lane minimum, whose dependency record is copied when it changes.
      seq += 1;
      const int par = seq & 1;
      if (tid == 0) {
        s_ntouch = 0;
        s_nrel = 0;
        s_ngl = 0;
      }
      {
        const uint32_t d = s_dirty[warp];
        if (d) {
          if ((d >> lane) & 1u) {
            mw = kInfBits;
            mk = INT_MAX;
#pragma unroll 4
            for (int q = tid; q < ng; q += kLazyThreads) {
              const long long w = gw[q];
              const int k = gk[q];
              if (lex_less(w, k, mw, mk)) {
                mw = w;
                mk = k;
              }
            }
          }
          __syncwarp();
          if (lane == 0) s_dirty[warp] = 0u;
        }
        const int src = warp_argmin(mw, mk);
        const long long w = __shfl_sync(0xFFFFFFFFu, mw, src);
        const int kk = w != kInfBits ? __shfl_sync(0xFFFFFFFFu, mk, src) : INT_MAX;
        PostStage &st = red[warp];
        if (VD) copy_wait();  // the record asked for in an earlier event
        __syncwarp();
        if (lane == 0) {
          st.w = w;
          st.k = kk;
          if (kk != cand_k) st.epoch = seq;
        }
        if (VD && kk != cand_k && w != kInfBits && lane < 3) copy16_async(&st.v + lane, r.net.vdep + 3 * (int64_t)kk + lane);
        cand_k = kk;
      }
      __syncthreads();
      if (warp == kPostWarp) {
        const long long w0 = lane < kLazyWarps ? red[lane].w : kInfBits;
        const int kk0 = lane < kLazyWarps ? red[lane].k : INT_MAX;
        const int src = warp_argmin(w0, kk0);
        const long long w = __shfl_sync(0xFFFFFFFFu, w0, src);
        const int kk = __shfl_sync(0xFFFFFFFFu, kk0, src);
        int4 v = make_int4(0, 0, 0, 0), rb = v, rl = v;
        double a = 0.0;
        if (w != kInfBits) {
          if (VD) {
            const PostStage &st = red[src];
            const int4 *rec = r.net.vdep + 3 * (int64_t)kk;
            const bool have = st.epoch != seq;
            v = have ? st.v : rec[0];
            rb = have ? st.rb : rec[1];
            rl = have ? st.rl : rec[2];
          }
          if (LL) a = CH[kk].a;
        }
        const int vw[4] = {v.x, v.y, v.z, v.w}, rbv[4] = {rb.x, rb.y, rb.z, rb.w}, rlv[4] = {rl.x, rl.y, rl.z, rl.w};
        if (lane < C) {
          const unsigned long long tag = mail_tag(seq);
          const uint32_t slot = map_rank(mb_local + (uint32_t)((par * kLazyMaxC + c) * sizeof(Mail)), lane);
          st_cluster(slot, (unsigned long long)w | tag);
          st_cluster(slot + 8, ((unsigned long long)seq << 32) | (uint32_t)kk);
          if (LL) st_cluster(slot + 16, (unsigned long long)dbits(a) | tag);
          if (VD) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              st_cluster(slot + 24 + 8 * i, ((unsigned long long)(uint32_t)rbv[i] << 32) | (uint32_t)vw[i] | tag);
            st_cluster(slot + 56, ((unsigned long long)(uint32_t)rlv[1] << 32) | (uint32_t)rlv[0] | tag);
            st_cluster(slot + 64, ((unsigned long long)(uint32_t)rlv[3] << 32) | (uint32_t)rlv[2] | tag);
          }
        }
        // While the posts travel: if this slice's candidate is the one that fires, the touched-
        // channel phase of every CTA starts by reading its reader lists.  Prefetch their lines
        // into L2 now (one CTA's candidate fires, so one CTA's prefetch is the useful one; the
        // others cost L2 traffic only), with the fired channel's own record, increment and group.
        if (VD && w != kInfBits) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (vpack_delta(vw[i]) == 0 || rlv[i] <= 0) continue;
            const uintptr_t b = (uintptr_t)(r.net.slist + rbv[i]) & ~(uintptr_t)127;
            const uintptr_t e = (uintptr_t)(r.net.slist + rbv[i] + rlv[i] - 1);
            for (uintptr_t p = b + (uintptr_t)lane * 128; p <= e; p += 32 * 128) prefetch_l2((const void *)p);
          }
          if (lane == 0) {
            prefetch_l2(CH + kk);
            prefetch_l2(ENX + kk);
            prefetch_l2(TAU + (kk & ~31));
            prefetch_l2(TAU + (kk & ~31) + 16);
          }
        }
      }
      if (warp == 0) {
        // wait (bounded) for every word of the C posts of this event
        bool ok = true;
        const unsigned long long tag = mail_tag(seq);
        long long it = 0;
        for (int i = lane; i < C * kMailWords && ok; i += 32) {
          const int wd = i % kMailWords;
          if ((wd == 2 && !LL) || (wd > 2 && !VD)) continue;
          const unsigned long long *p = &mbox[par][i / kMailWords].word[wd];
          for (;;) {
            const unsigned long long v = ld_mail(p);
            if (wd == 1 ? (unsigned)(v >> 32) == seq : (v >> 63) == (tag >> 63)) break;
            if (++it > L.spin_limit) {
              ok = false;
              break;
            }
            if (it > 4096) __nanosleep(32);  // a sleep lasts about a microsecond: only when something is amiss
          }
        }
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (lane == 0) s_ok = ok ? 1 : 0;
      }
      __syncthreads();
      // ---- 2. every thread takes the same decision from the C posts
      if (!s_ok) {
        status = RT_TRAJ_TIMEOUT;
        break;
      }
      constexpr unsigned long long kData = ~(1ull << 63);  // without the tag
      const long long pw = lane < C ? (long long)(ld_mail(&mbox[par][lane].word[0]) & kData) : kInfBits;
      const int pk = lane < C ? (int)(uint32_t)ld_mail(&mbox[par][lane].word[1]) : INT_MAX;
      const int qb = warp_argmin(pw, pk);
      const long long wmin = __shfl_sync(0xFFFFFFFFu, pw, qb);
      const int mu = __shfl_sync(0xFFFFFFFFu, pk, qb);
      if (wmin == kInfBits) {
        status = RT_TRAJ_ABSORBED;
        break;
      }
      if (wmin > tend_bits) {
        status = RT_TRAJ_TEND;
        break;
      }
      if (ev == r.max_events) {
        status = RT_TRAJ_MAX_EVENTS;
        break;
      }
      const unsigned long long *m = mbox[par][qb].word;
      int vw4[4], sp4[4], dl4[4], lb4[4], lo4[5];  // VD: changed species, their changes, their reader lists
      bool over = false;
      int vlen = 0;
      if (VD) {
        unpack(m, vw4, lb4, lo4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // unused entries are zero words behind the used ones
          const bool use = vpack_delta(vw4[i]) != 0;
          sp4[i] = use ? vpack_species(vw4[i]) : -1;
          dl4[i] = use ? vpack_delta(vw4[i]) : 0;
          if (use) over |= (int)((uint32_t)Xs[sp4[i]] + (uint32_t)dl4[i]) < 0;  // past INT_MAX it wraps below 0
        }
      } else {
        if (tid == 0) {
          const int vb = r.net.vptr[mu], ve = r.net.vptr[mu + 1];
          int n = 0, tot = 0;
          for (int i = vb; i < ve; ++i) {
            const int2 e = r.net.vlist[i];
            lists.vl[n] = e;
            lists.beg[n] = sptr[e.x];
            lists.ofs[n] = tot;
            tot += sptr[e.x + 1] - sptr[e.x];
            ++n;
          }
          lists.ofs[n] = tot;
          lists.vlen = n;
        }
        __syncthreads();
        vlen = lists.vlen;
        for (int i = 0; i < vlen; ++i) over |= (int)((uint32_t)Xs[lists.vl[i].x] + (uint32_t)lists.vl[i].y) < 0;
      }
      if (over) {
        status = RT_TRAJ_OVERFLOW;
        break;
      }
      const double tn = bitsd(wmin);
      if (c == 0 && gi < r.G && dbits(next_g) < wmin) {
        while (gi < r.G && dbits(next_g) < wmin) {
          record(gi, true);
          ++gi;
          next_g = __dmul_rn(__ll2double_rn(gi), r.sample_dt);
        }
      }
      t = tn;
      if (c == 0 && tid == 0) {
        trace_event(r.out, j, ev, mu, tn);
        if (LL) ll = __dadd_rn(ll, rt_ln(bitsd((int64_t)(ld_mail(m + 2) & kData))));
      }
      ++ev;
      // X after the event (Eq. 5); Xs itself is updated behind the next barrier
      auto xat = [&](int s) {
        int x = Xs[s];
        if (VD) {
#pragma unroll
          for (int i = 0; i < 4; ++i) x += sp4[i] == s ? dl4[i] : 0;
        } else {
          for (int i = 0; i < vlen; ++i) x += lists.vl[i].x == s ? lists.vl[i].y : 0;
        }
        return x;
      };
      // ---- 3. the touched channels of this slice: new a_k and tau_k
      // a touched channel, found in changed species li's reader list, as entry i of this event's list
      auto update = [&](int64_t k, int li, int i) {
        // one trip to memory for all three
        const int2 rd = r.net.rdesc[k];
        const double ck = r.net.c[k];
        ChanRec q = CH[k];
        // a channel reading two changed species is updated once, from its first list
        bool dup = false;
        if (VD) {
#pragma unroll
          for (int n = 0; n < 3; ++n) dup |= n < li && (rd.x == sp4[n] || (rd.y >= 0 && rd.y == sp4[n]));
        } else {
          for (int n = 0; n < li; ++n) dup |= rd.x == lists.vl[n].x || (rd.y >= 0 && rd.y == lists.vl[n].x);
        }
        if (dup) return;
        q.T = __dadd_rn(q.T, __dmul_rn(q.a, __dsub_rn(t, q.s)));
        q.s = t;
        q.a = propensity(rd, ck, xat);
        const double tau = lazy_tau(q.P, q.T, q.a, t);
        CH[k] = q;
        TAU[k] = tau;
        touch(k, dbits(tau), i >= 0 ? i : take_number(&s_ntouch));
      };
      if (warp < kFireTid / 32) {
        const int tot = VD ? lo4[4] : lists.ofs[vlen];
        for (int e = tid; e < tot; e += kFireTid) {
          int li = 0, at;
          if (VD) {
            at = entry(e, lb4, lo4, li);
          } else {
            while (e >= lists.ofs[li + 1]) ++li;
            at = lists.beg[li] + (e - lists.ofs[li]);
          }
          const int64_t k = r.net.slist[at];
          if (k < k0 || k >= k1 || k == mu) continue;
          if (L.compact) {  // the slice's channels, packed, for full warps below
            prefetch_l1(CH + k);
            prefetch_l1(r.net.rdesc + k);
            prefetch_l1(r.net.c + k);
            const int i = take_number(&s_ntouch);
            tk[i] = (int)k;
            tnext[i] = li;
          } else {
            update(k, li, -1);
          }
        }
      }
      if (L.compact) {
        __syncthreads();
        const int n = s_ntouch;
        if (warp < kFireTid / 32) {
          for (int i = tid; i < n; i += kFireTid) update(tk[i], tnext[i], i);
          // The slice whose candidate came second is the likeliest to fire next (its candidate unless the
          // firing slice's new minimum or a touched channel precedes it): the warps without a channel
          // bring what this slice would read for it from memory into L2.
          const int busy = min((n + 31) & ~31, kFireTid);
          if (VD && tid >= busy) {
            const int q2 = warp_argmin(lane == qb ? kInfBits : pw, lane == qb ? INT_MAX : pk);
            if (__shfl_sync(0xFFFFFFFFu, pw, q2) != kInfBits && q2 != qb) {
              int vw2[4], lb2[4], lo2[5], li;
              unpack(mbox[par][q2].word, vw2, lb2, lo2);
              for (int e = tid - busy; e < lo2[4]; e += kFireTid - busy) {
                const int64_t k = r.net.slist[entry(e, lb2, lo2, li)];
                if (k >= k0 && k < k1) {
                  prefetch_l2(CH + k);
                  prefetch_l2(TAU + (k & ~31));
                  prefetch_l2(TAU + (k & ~31) + 16);
                  prefetch_l2(r.net.rdesc + k);
                  prefetch_l2(r.net.c + k);
                }
              }
            }
          }
        }
      }
      if (tid == kFireTid && mu >= k0 && mu < k1) {
        // the fired channel: internal time up to the event, its next increment (drawn ahead,
        // Eq. 27; here only if it fired last in this slice too), new propensity and firing time
        ChanRec q = CH[mu];
        const int2 rd = r.net.rdesc[mu];
        const double ck = r.net.c[mu];
        const int32_t n = NK[mu] + 1;
        const double E = s_pend_k == mu ? exp1_draw(r.seed, g, (uint32_t)mu, (uint32_t)n, r.stream_id) : ENX[mu];
        NK[mu] = n;
        q.T = __dadd_rn(q.T, __dmul_rn(q.a, __dsub_rn(t, q.s)));
        q.s = t;
        q.P = __dadd_rn(q.P, E);
        q.a = propensity(rd, ck, xat);
        CH[mu] = q;
        const double tau = lazy_tau(q.P, q.T, q.a, t);
        TAU[mu] = tau;
        touch(mu, dbits(tau), L.compact ? L.cap - 1 : take_number(&s_ntouch));
      }
      if (warp == kPostWarp) {
        // the next increment of the channel this CTA fired last (Eq. 24, 27)
        if (lane == 0 && s_pend_k >= 0 && s_pend_k != mu)
          ENX[s_pend_k] = exp1_draw(r.seed, g, (uint32_t)s_pend_k, (uint32_t)(s_pend_n + 1), r.stream_id);
      }
      __syncthreads();
      if (warp == kPostWarp) {  // nothing reads Xs or the pending channel before the next barrier
        if (VD) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (lane == i && sp4[i] >= 0) Xs[sp4[i]] += dl4[i];  // species are distinct within one reaction
        } else if (lane < vlen) {
          Xs[lists.vl[lane].x] += lists.vl[lane].y;
        }
        if (lane == 31) {
          s_pend_k = mu >= k0 && mu < k1 ? mu : -1;
          if (mu >= k0 && mu < k1) s_pend_n = NK[mu];
        }
      }
      // ---- 4. group minima, one thread per touched group.  A group takes the smaller of its
      // previous minimum and its touched channels' minimum, unless its previous minimum channel was
      // touched and its tau grew: then every untouched channel may now be smaller, and the group is
      // reloaded below (its untouched channels from memory).  (If that channel's tau did not grow,
      // every untouched channel still lies above it.)
      const int ngl = s_ngl;
      for (int gi2 = tid; gi2 < ngl; gi2 += kLazyThreads) {
        const int q = glist[gi2];
        long long bw = kInfBits;
        int bk = INT_MAX;
        uint32_t bits = 0;
        bool hit = false;
        const int old_k = gk[q];
        const long long old_w = gw[q];
        for (int i = ghead[q]; i >= 0; i = tnext[i]) {
          const int k = tk[i];
          const long long w = tw[i];
          bits |= 1u << (k & 31);  // slices start at multiples of 32
          hit |= k == old_k && w > old_w;  // tau >= 0: bit patterns order like the values
          if (lex_less(w, k, bw, bk)) {
            bw = w;
            bk = k;
          }
        }
        ghead[q] = -1;
        if (hit) {
          const int ri = atomicAdd(&s_nrel, 1);
          rq[ri] = q;
          rcw[ri] = bw;
          rck[ri] = bk;
          rmask[ri] = bits;
        } else if (lex_less(bw, bk, old_w, old_k)) {
          set_group(q, bw, bk);
        }
      }
      __syncthreads();
      const int nrel = s_nrel;
      if (nrel) {
        for (int ri = warp; ri < nrel; ri += kLazyWarps) {
          const int q = rq[ri];
          const int64_t k = k0 + (int64_t)q * 32 + lane;
          const uint32_t bits = rmask[ri];
          const int first = __ffs((int)bits) - 1;  // a touched lane stands for all of them
          long long w = kInfBits;
          int kk = INT_MAX;
          if (k < k1 && !((bits >> lane) & 1u)) {
            w = dbits(__ldcg(TAU + k));
            kk = (int)k;
          } else if (lane == first) {
            w = rcw[ri];
            kk = rck[ri];
          }
          if (lane == warp_argmin(w, kk)) set_group(q, w, kk);
        }
        __syncthreads();
      }
    }
  }
  if (VD) copy_wait();

  // ---- finalise
  const bool known = status == RT_TRAJ_TEND || status == RT_TRAJ_ABSORBED;
  if (c == 0)
    for (; gi < r.G; ++gi) record(gi, known);
  if (L.want_T && !bad) {
    // every channel's internal time up to the end of the run
    const double tf = (known && L.tend_finite) ? r.t_end : t;
    for (int64_t k = k0 + tid; k < k1; k += blockDim.x) {
      ChanRec q = CH[k];
      q.T = __dadd_rn(q.T, __dmul_rn(q.a, __dsub_rn(tf, q.s)));
      q.s = tf;
      CH[k] = q;
    }
  }
  if (r.out.t_internal_dev)
    for (int64_t k = k0 + tid; k < k1; k += blockDim.x) r.out.t_internal_dev[j * M + k] = CH[k].T;
  if (r.out.counts_dev)
    for (int64_t k = k0 + tid; k < k1; k += blockDim.x) r.out.counts_dev[j * M + k] = NK[k];
  __threadfence();
  cluster.sync();  // every slice is final; no CTA posts into a mailbox after this point
  if (LL && c == 0 && tid == 0) {
    double sT = 0.0;
    if (!bad)
      for (int k = 0; k < M; ++k) sT = __dadd_rn(sT, __ldcg(&CH[k].T));
    r.out.loglik_dev[j] = bad ? __longlong_as_double(0x7FF8000000000000ll) : __dsub_rn(ll, sT);
  }
  if (c == 0) {
    trace_tail(r.out, j, ev, tid, blockDim.x);
    if (r.out.x_final_dev)
      for (int s = tid; s < N; s += blockDim.x) r.out.x_final_dev[j * N + s] = Xs[s];
    if (tid == 0) {
      if (r.out.n_events_dev) r.out.n_events_dev[j] = ev;
      if (r.out.status_dev) r.out.status_dev[j] = status;
      if (r.out.t_last_dev) r.out.t_last_dev[j] = t;
    }
  }
}

// ----------------------------------------------------------------------------------
// host side
// ----------------------------------------------------------------------------------

static int64_t round_up_l(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

struct LazyPlan {
  int C;
  int64_t chunk, Ms;
  size_t off_CH, off_TAU, off_ENX, off_NK, total;
  size_t smem;
  int sptr_smem;
  int cap;
  int compact;
};

static LazyPlan plan_lazy(const DevNet &net, int max_dependents, int64_t n_traj, int C, size_t smem_budget) {
  LazyPlan p;
  p.C = C;
  p.chunk = round_up_l((net.M + C - 1) / C, 32);
  p.Ms = p.chunk * C;
  const int64_t rows = n_traj > 0 ? n_traj : 1;
  size_t off = 0;
  p.off_CH = off; off += (size_t)rows * p.Ms * sizeof(ChanRec);
  p.off_TAU = off; off += (size_t)rows * p.Ms * 8;
  p.off_ENX = off; off += (size_t)rows * p.Ms * 8;
  p.off_NK = off; off += (size_t)round_up_l(rows * p.Ms * 4, 256);
  p.total = off;
  const int ng = (int)(p.chunk / 32);
  // touched channels of one event in one slice: at most the fired channel and the readers of
  // the species it changes (max_dependents counts them with multiplicity); with each channel once
  // per changed reactant if that list fits too (the fired channel in the last entry)
  // gw, gk, ghead per group; tw, rcw, tk, tnext, glist, rq, rck, rmask per touched channel; X
  auto size = [&](int64_t cap) {
    return (size_t)ng * (8 + 4 + 4) + (size_t)cap * (8 + 8 + 4 + 4 + 4 + 4 + 4 + 4) + (size_t)net.N * 4;
  };
  const int64_t once = std::min<int64_t>(p.chunk, (int64_t)max_dependents + 1);
  const int64_t twice = std::min<int64_t>(2 * p.chunk, (int64_t)max_dependents) + 1;
  p.compact = size(twice) <= smem_budget ? 1 : 0;
  p.cap = (int)(p.compact ? twice : once);
  const size_t base = size(p.cap);
  // the species offsets are read only where reactions have no dependency records
  p.sptr_smem = !net.vdep && base + (size_t)(net.N + 1) * 4 <= smem_budget ? 1 : 0;
  p.smem = base + (p.sptr_smem ? (size_t)(net.N + 1) * 4 : 0);
  return p;
}

constexpr size_t kLazySmemBudget = 200 * 1024;

typedef void (*LazyKernel)(const LazyArgs);
static LazyKernel lazy_kernel(bool ll, bool vd) {
  return ll ? (vd ? k_lazy<true, true> : k_lazy<true, false>) : (vd ? k_lazy<false, true> : k_lazy<false, false>);
}

// Clusters of C CTAs of the lazy kernel that can be resident at once (0: does not fit).
static int lazy_active_clusters(const LazyPlan &p, bool ll, bool vd) {
  if (p.smem > kLazySmemBudget) return 0;
  auto kern = lazy_kernel(ll, vd);
  if (raise_smem_limit((const void *)kern, p.smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (p.C > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.C);
  cfg.blockDim = dim3(kLazyThreads);
  cfg.dynamicSmemBytes = p.smem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)p.C;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, (void *)kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

// CTAs per trajectory: the largest power of two (<= 8, and <= M / 32) with which every
// trajectory is resident at once, else the one that keeps the most trajectories resident.
static int choose_lazy_C(const DevNet &net, int maxdep, int64_t n_traj, int requested, bool ll) {
  if (requested > 0) return requested;
  int best = 1;
  int64_t best_res = -1;
  for (int C = 8; C >= 1; C /= 2) {
    if (C > 1 && (int64_t)net.M < 32 * (int64_t)C) continue;
    const int act = lazy_active_clusters(plan_lazy(net, maxdep, n_traj, C, kLazySmemBudget), ll, net.vdep != nullptr);
    if (act <= 0) continue;
    if (act >= n_traj) return C;
    const int64_t res = (int64_t)act;
    if (res > best_res) {
      best_res = res;
      best = C;
    }
  }
  return best;
}

size_t lazy_workspace_bytes(const DevNet &net, int max_dependents, int64_t n_traj, int ctas_per_traj) {
  int C = 0;
  for (int ll = 0; ll < 2; ++ll) C = std::max(C, choose_lazy_C(net, max_dependents, n_traj, ctas_per_traj, ll));
  size_t b = 0;
  for (int c2 = 1; c2 <= C; c2 *= 2) b = std::max(b, plan_lazy(net, max_dependents, n_traj, c2, kLazySmemBudget).total);
  return std::max(b, plan_lazy(net, max_dependents, n_traj, C, kLazySmemBudget).total);
}

int launch_lazy_mapping(const RunArgs &a, int max_dependents, int ctas_per_traj, void *ws, size_t ws_bytes,
                        cudaStream_t s) {
  if (a.n_traj == 0) return RT_OK;
  if (a.net.max_vlen > kLazyMaxVlen)
    return set_error(RT_ERR_UNSUPPORTED, "absolute-time form: a reaction changes %d species (at most %d)",
                     a.net.max_vlen, kLazyMaxVlen);
  const bool ll = a.out.loglik_dev != nullptr;
  const int C = choose_lazy_C(a.net, max_dependents, a.n_traj, ctas_per_traj, ll);
  if (C < 1 || C > kLazyMaxC || (C & (C - 1)))
    return set_error(RT_ERR_INVALID_ARG, "absolute-time form: ctas_per_traj must be a power of two <= %d", kLazyMaxC);
  const LazyPlan p = plan_lazy(a.net, max_dependents, a.n_traj, C, kLazySmemBudget);
  if (p.smem > kLazySmemBudget)
    return set_error(RT_ERR_UNSUPPORTED, "absolute-time form: %d species and %lld channels per CTA do not fit in "
                     "shared memory (%zu bytes)", a.net.N, (long long)p.chunk, p.smem);
  if (!ws || ws_bytes < p.total)
    return set_error(RT_ERR_OOM, "absolute-time form needs %zu bytes of workspace (got %zu)", p.total, ws_bytes);
  if (((uintptr_t)ws & 255) != 0) return set_error(RT_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
  // every check before the first enqueued operation
  if (a.n_traj * C > INT_MAX) return set_error(RT_ERR_UNSUPPORTED, "absolute-time form: too many trajectories for one launch");
  if (lazy_active_clusters(p, ll, a.net.vdep != nullptr) < 1)
    return set_error(RT_ERR_UNSUPPORTED, "absolute-time form: a cluster of %d CTAs cannot be resident", C);
  char *w = (char *)ws;
  LazyArgs L;
  L.r = a;
  L.C = C;
  L.Ms = p.Ms;
  L.chunk = p.chunk;
  L.CH = (ChanRec *)(w + p.off_CH);
  L.TAU = (double *)(w + p.off_TAU);
  L.ENX = (double *)(w + p.off_ENX);
  L.NK = (int32_t *)(w + p.off_NK);
  L.cap = p.cap;
  L.compact = p.compact;
  L.sptr_smem = p.sptr_smem;
  L.tend_finite = std::isfinite(a.t_end) ? 1 : 0;
  L.want_T = (a.out.t_internal_dev || a.out.loglik_dev) ? 1 : 0;
  // polls before a trajectory gives up, with a sleep of about a microsecond each after the first 4096: some 20 s
  long long spin = 20000000;
  if (const char *env = getenv("RT_DEBUG_SPIN_LIMIT")) spin = atoll(env);
  L.spin_limit = spin;
  k_lazy_init<<<152 * 8, 256, 0, s>>>(L);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return set_error(RT_ERR_CUDA, "init launch: %s", cudaGetErrorString(e));
  auto kern = lazy_kernel(ll, a.net.vdep != nullptr);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_traj * C));
  cfg.blockDim = dim3(kLazyThreads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)C;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, L);
  if (e != cudaSuccess) return set_error(RT_ERR_CUDA, "absolute-time kernel launch: %s", cudaGetErrorString(e));
  return RT_OK;
}

}  // namespace rt

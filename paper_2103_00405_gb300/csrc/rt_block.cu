// rt_block.cu -- one thread block per trajectory (RT_MAP_BLOCK): the single-network
// kernel around block_trajectory (rt_traj_block.cuh), for networks of up to
// 8 * block_threads reactions: T in registers, propensities and float bounds in shared
// memory (in local memory where many species leave no room), P and the next increments in
// local memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "rt_traj_block.cuh"

namespace rt {

// 64 registers: two resident blocks of 512 threads per SM, or more smaller ones.
template <int R, bool LL, bool SM>
__global__ void __launch_bounds__(512, 2) k_ens_block(const RunArgs A, const int tend_finite) {
  extern __shared__ __align__(16) unsigned char smem[];
  const BlockScratch S = carve_block_scratch(smem, SM ? block_state_bytes(A.net.M, blockDim.x) : 0, A.net.M, A.net.N,
                                             blockDim.x);
  const BlockNet net{A.net.M, A.net.N, A.net.rdesc, A.net.c, A.net.vptr, A.net.vlist, A.net.dptr, A.net.dlist};
  for (int64_t j = blockIdx.x; j < A.n_traj; j += gridDim.x) block_trajectory<R, LL, SM>(A, net, S, j, tend_finite);
}

constexpr size_t kBlockSmemMax = 226 * 1024;  // of the 227 KB a block can have

int block_mapping_max_m() { return 4096; }

template <int R, bool SM>
static cudaError_t launch_r(const RunArgs &a, int B, cudaStream_t s, int tf) {
  const size_t smem = block_scratch_bytes(a.net.M, a.net.N, B) + (SM ? block_state_bytes(a.net.M, B) : 0);
  auto kern = a.out.loglik_dev ? k_ens_block<R, true, SM> : k_ens_block<R, false, SM>;
  raise_smem_limit((const void *)kern, smem);
  int per_sm = 0, dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, B, smem);
  const int64_t grid = std::min<int64_t>(a.n_traj, (int64_t)std::max(1, per_sm) * sms);
  kern<<<(unsigned)grid, B, smem, s>>>(a, tf);
  return cudaGetLastError();
}

// The fewest threads of a block left to the library: one for eight channels.
static int fewest_threads(int M) { return std::min(512, std::max(64, ((M + 7) / 8 + 31) / 32 * 32)); }

// Threads per trajectory: between one for eight channels and one each, as many as let the SM's share of
// the trajectories be resident at 64 registers (1024 threads).  A block with few slots per thread takes
// fewer instructions one after the other per event; with many, more trajectories share the SM.
static int choose_threads(int M, int64_t n_traj) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t per_sm = std::max<int64_t>(1, (n_traj + sms - 1) / std::max(1, sms));
  const int hi = std::min(512, (M + 31) / 32 * 32);
  const int fit = (int)std::max<int64_t>(0, 1024 / per_sm) / 32 * 32;
  return std::max(fewest_threads(M), std::min(hi, fit));
}

int launch_block_mapping(const RunArgs &a, int block_threads, cudaStream_t s) {
  if (a.n_traj == 0) return RT_OK;
  const int M = a.net.M;
  int B = block_threads;
  if (B <= 0) B = choose_threads(M, a.n_traj);
  if (B % 32 || B > 512) return set_error(RT_ERR_INVALID_ARG, "block mapping: block_threads must be a multiple of 32 <= 512");
  const int R = (M + B - 1) / B;
  if (R > 8) return set_error(RT_ERR_UNSUPPORTED, "block mapping supports M <= 8 * block_threads (M = %d)", M);
  // What is refused: more than 200 KB for X, the counts, the bitmap and an allowance of 24 bytes a warp and 8
  // a thread.  A block size left to the library is taken as the smallest, so that the number of trajectories
  // does not decide; the scratch that is launched (40 bytes a thread) is at most 20 KB more and fits.
  const int Bf = block_threads > 0 ? B : fewest_threads(M);
  if ((size_t)a.net.N * 4 + (size_t)M * 4 + (size_t)((M + 31) / 32) * 4 + (size_t)(Bf / 32) * 24 + (size_t)Bf * 8 + 96 >
      200 * 1024)
    return set_error(RT_ERR_UNSUPPORTED, "block mapping: %d species do not fit in shared memory", a.net.N);
  const int tf = std::isfinite(a.t_end) ? 1 : 0;
  cudaError_t e;
  if (block_state_bytes(M, B) + block_scratch_bytes(M, a.net.N, B) > kBlockSmemMax) {
    e = launch_r<8, false>(a, B, s, tf);  // many species leave no room for the state
  } else {
    switch (R) {
      case 1: e = launch_r<1, true>(a, B, s, tf); break;
      case 2: e = launch_r<2, true>(a, B, s, tf); break;
      case 3: e = launch_r<3, true>(a, B, s, tf); break;
      case 4: e = launch_r<4, true>(a, B, s, tf); break;
      case 5: e = launch_r<5, true>(a, B, s, tf); break;
      case 6: e = launch_r<6, true>(a, B, s, tf); break;
      case 7: e = launch_r<7, true>(a, B, s, tf); break;
      default: e = launch_r<8, true>(a, B, s, tf); break;
    }
  }
  if (e != cudaSuccess) return set_error(RT_ERR_CUDA, "block kernel launch: %s", cudaGetErrorString(e));
  return RT_OK;
}

}  // namespace rt

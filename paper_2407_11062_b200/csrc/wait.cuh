// Bounded waits on mbarriers, and the status word of the kernels that gave one up.  Included by every file with kernels
// that wait: each gets a status word, a self-test kernel and a read-out of its own.
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace eqat {
namespace {

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s per wait

__device__ int g_wait_status[2];       // [0] = eqat_status, [1] = WaitSite

// Waits for an mbarrier phase, for at most `limit_ns`; false once the limit has passed or `*abort` says that another wait
// of the CTA has run out.  `sleep_ns` > 0 backs off between polls, so that a role with nothing to do for a long time leaves
// the issue slots to the warps that are working; latency-critical waits pass 0.  CLUSTER: the barrier is also signalled from
// another CTA.
template <bool CLUSTER = false>
__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, volatile int* abort, int site,
                                             uint32_t sleep_ns = 0, uint64_t limit_ns = kWaitLimitNs) {
  auto ready = [&] { return CLUSTER ? ptx::mbar_try_wait_cluster(bar, parity) : ptx::mbar_try_wait(bar, parity); };
  if (ready()) return true;
  uint64_t t0 = 0;
  uint32_t n = 0;
  while (!ready()) {
    if (sleep_ns != 0) __nanosleep(sleep_ns);
    if ((++n & 31u) == 0u) {
      if (*abort) return false;
      const uint64_t t = ptx::globaltimer_ns();
      if (t0 == 0) t0 = t;                               // the clock is read only by waits that turn out long
      if (t - t0 > limit_ns) {
        *abort = 1;
        atomicExch(&g_wait_status[1], site);
        atomicExch(&g_wait_status[0], (int)EQAT_ERR_TIMEOUT);
        return false;
      }
    }
  }
  return true;
}

// Waits of a whole warp: it goes on or gives up together.  The lanes of a warp may see the abort flag change, or the limit
// pass, one earlier than the other, and what follows (elect.sync, shuffles, tcgen05) wants all of them.
// (Loops that issue MMAs vote after the issue instead, off its path.)
template <bool CLUSTER = false>
__device__ __forceinline__ bool bounded_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort, int site,
                                                  uint32_t sleep_ns = 0) {
  return __all_sync(0xFFFFFFFFu, bounded_wait<CLUSTER>(bar, parity, abort, site, sleep_ns));
}

// The same vote as a ballot.  With __all_sync the compiler knows the exit of the loop to be uniform and keeps its counters in
// uniform registers, which cost the MMA warp of the GEMM kernels 0.5 us (ds of 512 x 512, 300 tokens 7.7 -> 8.2 us, of 4096
// x 4096 24.1 -> 25.5 us); the ballot costs them nothing.  The weight-row kernels lose 0.5 % with __all_sync, 1 % with this.
__device__ __forceinline__ bool warp_agrees(bool got) { return got & (__ballot_sync(0xFFFFFFFFu, got) == 0xFFFFFFFFu); }

// The give-up path alone (abort flag, status word, normal return), without any copy or tensor-memory state around it: one
// warp, a barrier nothing signals, a short limit.
__global__ void wait_expiry_kernel(uint64_t limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_word;
  if (threadIdx.x == 0) {
    ptx::mbar_init(ptx::smem_addr(&bar), 1);
    abort_word = 0;
    ptx::fence_mbar_init();
  }
  __syncthreads();
  (void)bounded_wait(ptx::smem_addr(&bar), 0u, &abort_word, WAIT_SELFTEST, 0, limit_ns);
}

inline int launch_wait_expiry(cudaStream_t st) {
  wait_expiry_kernel<<<1, 32, 0, st>>>(1000000ull);      // 1 ms
  return launch_status();
}

// Reads and clears the status word; synchronises.
inline int read_wait_status(int* status, int* detail) {
  int h[2] = {0, 0};
  if (cudaDeviceSynchronize() != cudaSuccess) return EQAT_ERR_CUDA;
  if (cudaMemcpyFromSymbol(h, g_wait_status, sizeof(h)) != cudaSuccess) return EQAT_ERR_CUDA;
  const int zero[2] = {0, 0};
  if (cudaMemcpyToSymbol(g_wait_status, zero, sizeof(zero)) != cudaSuccess) return EQAT_ERR_CUDA;
  *status = h[0];
  *detail = h[1];
  return EQAT_OK;
}

}  // namespace
}  // namespace eqat

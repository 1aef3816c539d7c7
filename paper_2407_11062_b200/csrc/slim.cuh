// Host launcher of the packed forward for a few tokens on weight-row tiles (arguments already validated).
#pragma once
#include <cuda_runtime.h>
#include "eqat.h"

namespace eqat {

// Launch shape, and the time it is expected to take.
struct SlimPlan {
  int nt, nd;                // token columns / 16 per tile, accumulators per run of 128 codes
  int token_tiles, split;    // split = CTAs of a cluster, over K
  int groups;                // quantisation groups of a row, the most that one CTA's slice touches
  double us;                 // 0: the problem does not fit
};
// True when the weight-row kernel is the one to take for this packed forward on a device of `sms` SMs, and how.
bool slim_fwd_applies(const eqat_desc& d, int sms, SlimPlan& plan);
// Y[T,out] = X[T,in] * dequant(Wq)^T
int launch_slim_fwd(const eqat_desc& d, const eqat_bf16* X, const uint8_t* Wq, const eqat_fp16* s16, const void* zq,
                    eqat_bf16* Y, const SlimPlan& plan, cudaStream_t st);

// Self-test of the kernel's bounded wait (one warp, 1 ms, a barrier nothing signals).
int launch_wait_expiry_slim(cudaStream_t st);
// Reads and clears the status word ({status, wait site}); synchronises.
int read_slim_status(int* status, int* detail);

}  // namespace eqat

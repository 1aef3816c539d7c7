// Host launcher of the packed forward for prompts on weight-row tiles (arguments already validated).
#pragma once
#include <cuda_runtime.h>
#include "eqat.h"

namespace eqat {

struct WidePlan {
  int tn, token_tiles;       // tokens per tile
  int split;                 // pairs of CTAs per cluster, over K
  int first_pairs;           // pairs of row tiles that are computed so; the others, in a launch of their own,
  int rest_split;            // with this split
  double us;                 // expected time; 0: the problem does not fit
};
// True when the kernel is the one to take for this packed forward, and how: on the current device (sms = 0), or on one of
// `sms` SMs that are grouped like a B200's.
bool wide_fwd_applies(const eqat_desc& d, int sms, WidePlan& plan);
// Y[T,out] = X[T,in] * dequant(Wq)^T
int launch_wide_fwd(const eqat_desc& d, const eqat_bf16* X, const uint8_t* Wq, const eqat_fp16* s16, const void* zq,
                    eqat_bf16* Y, const WidePlan& plan, cudaStream_t st);

// Self-test of the kernel's bounded wait (one warp, 1 ms, a barrier nothing signals).
int launch_wait_expiry_wide(cudaStream_t st);
// Reads and clears the status word ({status, wait site}); synchronises.
int read_wide_status(int* status, int* detail);

}  // namespace eqat

// Host launcher of the packed-weight matrix-vector forward (arguments already validated).
#pragma once
#include <cuda_runtime.h>
#include "eqat.h"

namespace eqat {

// How the few-token kernel would take a problem: launches over slices of `slice` tokens (0: not at all), and the
// expected time.
struct FewTokenPlan {
  int launches, slice;
  double us;
};
FewTokenPlan packed_gemv_plan(const eqat_desc& d);

// True where every batch of up to sixteen tokens goes through this kernel, so that a token gives the same bits alone and in
// any of them: weights of less than 3 MB of codes, rows of 1024 to 4096 columns, groups of at least 64.
bool packed_gemv_keeps_bits(const eqat_desc& d);
// True when the few-token kernel handles this problem: groups of at least 64 elements and tokens whose staged activations
// fit in the shared memory of a CTA, so that one launch takes them all, or the range above (two launches).  Where the tokens
// need more launches the weight-row kernel is faster on every shape and fits wherever this one does.
bool packed_gemv_applies(const eqat_desc& d);
// Y[T,out] = X[T,in] * dequant(Wq)^T for a problem packed_gemv_applies() accepted
int launch_packed_gemv(const eqat_desc& d, const eqat_bf16* X, const uint8_t* Wq, const eqat_fp16* s16,
                       const void* zq, eqat_bf16* Y, cudaStream_t st);

// Self-test of the matrix-vector kernel's bounded wait (one warp, 1 ms, a barrier nothing signals).
int launch_wait_expiry_gemv(cudaStream_t st);
// Reads and clears the status word of the matrix-vector kernels ({status, wait site}); synchronises.
int read_gemv_status(int* status, int* detail);

}  // namespace eqat

// firp_topb_static: the top-B of logits rows for callers that must not allocate device memory.  (The paper has no
// counterpart.)
#include <cstdio>

#include "../../include/firp.h"
#include "firp_kernels.cuh"

extern "C" int firp_topb_static(const float *d_logits, int32_t rows, int32_t vocab, int32_t b, int32_t *d_ids,
                                float *d_vals, void *stream) {
  if (!d_logits || !d_ids || !d_vals || rows < 1 || vocab < 1 || b < 1 || b > firp::kMaxTopB) {
    fprintf(stderr, "firp_topb_static: NULL pointer, or rows / vocab / b out of range (b must be 1..%d)\n", firp::kMaxTopB);
    return FIRP_ERR_BAD_ARG;
  }
  // The limit of the ABI, counted in 2048-logit segments (in 64 bits: vocab + 2047 would wrap for a vocab next to
  // INT32_MAX).  The selection itself keeps nothing in device memory.
  const long long slots = (long long)rows * (((long long)vocab + 2047) / 2048);
  if (slots > FIRP_TOPB_STATIC_MAX_SLOTS) {
    fprintf(stderr, "firp_topb_static: rows * ceil(vocab / 2048) = %lld exceeds the limit of %d slots\n", slots,
            FIRP_TOPB_STATIC_MAX_SLOTS);
    return FIRP_ERR_CAPACITY;
  }
  firp::launch_topb(d_logits, rows, vocab, b, d_ids, d_vals, true, (cudaStream_t)stream);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    fprintf(stderr, "firp_topb_static: launch failed: %s\n", cudaGetErrorString(e));
    return FIRP_ERR_CUDA;
  }
  return FIRP_OK;
}

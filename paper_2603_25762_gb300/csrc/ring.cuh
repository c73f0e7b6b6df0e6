// Uses of an operand ring by the producer of the multi-step kernel (bsb_run.cu).  Uses are
// numbered in the order of the copies; use n takes slot n % st, phase n / st.  Before the CTA
// exits the latest copy into every slot must have landed, also when the producer gave up
// part-way through a batch of copies that its lanes issue side by side.
// Plain C++ (no CUDA types), so a host compiler checks it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define QH_RING_FN __host__ __device__ __forceinline__
#else
#define QH_RING_FN static inline
#endif

namespace qh {

// The latest use of the slot that use q + l takes (0 <= l < st): uses 0 .. q - 1 were all
// issued, and of the batch from q on those whose bit in `part` is set.  False: none.
QH_RING_FN bool ring_last_use(uint32_t q, uint32_t part, uint32_t l, uint32_t st, uint32_t* use) {
  if ((part >> l) & 1u) {
    *use = q + l;
    return true;
  }
  *use = q + l - st;
  return q + l >= st;
}

}  // namespace qh

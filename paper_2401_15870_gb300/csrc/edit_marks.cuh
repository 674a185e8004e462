// edit_marks.cuh -- what the row edit (batch.cu, k_edit_long) keeps per old
// element of a chunk: one bit that says whether the batch deletes it, and a
// counter of what changes the shift in front of it (+1 for every insertion that
// falls between it and the element before, -1 when the element before is
// deleted).  An element's shift is the prefix sum of the counters up to its own.
//
// The two are kept apart: a counter takes any number of insertions a row can
// hold (ids are below 2^31), so no count may stand for "deleted".
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define EDITMARK_FN __host__ __device__ __forceinline__
#else
#define EDITMARK_FN inline
#endif

namespace editmarks {

// old element i is deleted: those behind it move down by one.  shift: the
// chunk's elements and one more; dead: a bit per element
EDITMARK_FN void mark_deleted(int32_t* shift, uint32_t* dead, int32_t i) {
#if defined(__CUDA_ARCH__)
  atomicOr(dead + (i >> 5), 1u << (i & 31));
  atomicAdd(shift + i + 1, -1);
#else
  dead[i >> 5] |= 1u << (i & 31);
  shift[i + 1] -= 1;
#endif
}

// k insertions in front of old element i
EDITMARK_FN void mark_inserted(int32_t* shift, int32_t i, int32_t k) {
#if defined(__CUDA_ARCH__)
  atomicAdd(shift + i, k);
#else
  shift[i] += k;
#endif
}

EDITMARK_FN bool is_deleted(const uint32_t* dead, int32_t i) { return (dead[i >> 5] >> (i & 31)) & 1u; }

}  // namespace editmarks

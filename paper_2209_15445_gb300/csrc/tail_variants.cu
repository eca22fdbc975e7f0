// The tail kernels with chords (variant 1) and with the step-length histogram (4, and 12 in the
// field).
#include <cuda_runtime.h>

#include "layout.h"
#include "tail.cuh"

namespace adept {

template <class R>
static const void* by_variant(int variant) {
  if (variant & 1) return (const void*)k_tail<R, 0, 1>;
  return (variant & 8) ? (const void*)k_tail<R, 4, 12> : (const void*)k_tail<R, 4, 4>;
}

const void* tail_variant_fn(int precision, int variant) {
  return precision ? by_variant<float>(variant) : by_variant<double>(variant);
}

}  // namespace adept

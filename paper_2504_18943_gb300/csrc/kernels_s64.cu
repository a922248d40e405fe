// Small levels in one launch, for 64-bit characteristic-sequence words.
#include "lsyn_small.cuh"

namespace lsyn {
template struct SmallKernels<uint64_t>;
}  // namespace lsyn

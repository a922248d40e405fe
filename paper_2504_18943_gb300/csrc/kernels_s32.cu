// Small levels in one launch, for 32-bit characteristic-sequence words.
#include "lsyn_small.cuh"

namespace lsyn {
template struct SmallKernels<uint32_t>;
}  // namespace lsyn

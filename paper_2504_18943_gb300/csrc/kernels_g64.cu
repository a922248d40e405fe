// Group kernels (matrices above 512 bytes) for 64-bit characteristic-sequence words.
#include "lsyn_group.cuh"

namespace lsyn {
template struct GroupKernels<uint64_t>;
}  // namespace lsyn

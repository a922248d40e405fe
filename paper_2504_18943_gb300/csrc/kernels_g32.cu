// Group kernels (matrices above 512 bytes) for 32-bit characteristic-sequence words.
#include "lsyn_group.cuh"

namespace lsyn {
template struct GroupKernels<uint32_t>;
}  // namespace lsyn

// Path-A level kernels (matrices of at most 128 bytes) for 32-bit characteristic-sequence words.
#include "lsyn_lanes.cuh"

namespace lsyn {
template struct LaneKernels<uint32_t>;
}  // namespace lsyn

// Path-A level kernels (matrices of at most 128 bytes) for 64-bit characteristic-sequence words.
#include "lsyn_lanes.cuh"

namespace lsyn {
template struct LaneKernels<uint64_t>;
}  // namespace lsyn

// Forward projector kernel: 3 j-blur strip(s) per thread, radii up to kMaxR.
#include "forward.cuh"

namespace spect {
template cudaError_t forward_launch_ipt<3, true>(const ForwardArgs&, cudaStream_t);
template int forward_occupancy_ipt<3, true>(int, size_t);
}  // namespace spect

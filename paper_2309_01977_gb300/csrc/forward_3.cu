// Forward projector kernel: 2 j-blur strip(s) per thread, radii up to kMaxR.
#include "forward.cuh"

namespace spect {
template cudaError_t forward_launch_ipt<2, true>(const ForwardArgs&, cudaStream_t);
template int forward_occupancy_ipt<2, true>(int, size_t);
}  // namespace spect
